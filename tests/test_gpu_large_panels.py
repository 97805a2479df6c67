"""The Householder panel's digit form at the orders where its shared memory decides (GPU only): with
16 blocks a matrix, column and digits side by side up to n = 2561, the column in the digits' space
up to n = 3649, the FP64 form beyond.  Each order runs the form it should (the digit form has a
stage of its own) on a well-conditioned pencil; all eigenpairs by residual and orthonormality.
Batches take other cluster sizes (16 matrices: 8 blocks each) and agree with single matrices."""
import pytest

from tests.gpu_helpers import TOL_EPS, TOL_ORTH, TOL_RES

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _pencil(n, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    G = torch.randn((n, n), generator=g, dtype=torch.complex128, device=DEV)
    H = (G + G.mH) / (2.0 * n ** 0.5)
    d = 0.5 + torch.rand(n, generator=g, dtype=torch.float64, device=DEV)
    u = torch.randn((n, 4), generator=g, dtype=torch.complex128, device=DEV) / n ** 0.5
    return H, torch.diag(d).to(H.dtype) + u @ u.mH


def _context():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_4247_gb300.nao import Context
    ctx = Context(0)
    ctx.nao_profile_enable(True)
    return ctx


@pytest.mark.parametrize("mixed", [False, True], ids=["fp64", "mixed"])
@pytest.mark.parametrize("n,digits", [(2561, True), (2562, True), (3104, True), (3649, True), (3650, False)])
def test_form_at_the_limits(n, digits, mixed):
    from paper_1402_4247_gb300.nao import NAO_FP64, NAO_MIXED_BF16X3
    ctx = _context()
    H, S = _pencil(n, n)
    # two Ritz sweeps bring the mixed mode's vectors to the FP64 bounds
    ctx.nao_set_refinement(2 if mixed else 0)
    eps, C, m, st = ctx.nao_gen_eig(H[None], S[None], precision=NAO_MIXED_BF16X3 if mixed else NAO_FP64)
    torch.cuda.synchronize()
    assert int(st[0]) == 0 and int(m[0]) == n
    assert ("hetrd_digits" in ctx.nao_profile_read()) == digits
    ctx.close()
    e, c = eps[0], C[0]
    assert bool((e[1:] >= e[:-1]).all())
    res = torch.linalg.norm(H @ c - (S @ c) * e[None, :]) / (n * float(e.abs().max()))
    assert float(res) <= TOL_RES
    assert float((c.mH @ S @ c - torch.eye(n, dtype=c.dtype, device=DEV)).abs().max()) <= TOL_ORTH


@pytest.mark.parametrize("n,P", [(2700, 3), (2562, 16)])
def test_batches_agree_with_single_matrices(n, P):
    ctx = _context()
    two = [_pencil(n, 50 + i) for i in range(2)]
    single = [ctx.nao_gen_eig(H[None], S[None], want_vectors=False)[0][0] for H, S in two]
    H = torch.stack([two[p % 2][0] for p in range(P)])
    S = torch.stack([two[p % 2][1] for p in range(P)])
    eps, _, m, st = ctx.nao_gen_eig(H, S, want_vectors=False)
    torch.cuda.synchronize()
    assert int(st.abs().sum()) == 0 and bool((m == n).all())
    assert "hetrd_digits" in ctx.nao_profile_read()
    ctx.close()
    for p in range(P):
        ref = single[p % 2]
        assert float((eps[p] - ref).abs().max()) <= TOL_EPS * float(ref.abs().max())
