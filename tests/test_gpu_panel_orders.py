"""The Householder panel over its launch shapes (GPU only): orders at the edges of its 16-row tiles
and 32-column panels, with few problems (many blocks share a matrix) and many (one block each),
in FP64 and mixed precision; eigenvalues against LAPACK, residual and orthonormality at the
parity bounds."""
import numpy as np
import pytest

from paper_1402_4247_gb300 import synth
from tests.gpu_helpers import TOL_EPS, TOL_ORTH, TOL_RES

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("precision", [0, 2], ids=["fp64", "mixed"])
@pytest.mark.parametrize("n,P", [(2, 3), (3, 1), (16, 2), (17, 1), (18, 160), (33, 1), (34, 7), (48, 40), (49, 2), (65, 1),
                                 (100, 30), (145, 1), (145, 160), (260, 1), (260, 90), (275, 153), (530, 2)])
def test_panel_shapes(n, P, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_4247_gb300.nao import Context
    rng = np.random.Generator(np.random.PCG64(9000 + 31 * n + P))
    base = [synth.random_hermitian_pair(rng, n, cond=30.0) for _ in range(min(P, 4))]
    H = torch.from_numpy(np.stack([base[p % len(base)][0] for p in range(P)])).to(DEV)
    S = torch.from_numpy(np.stack([base[p % len(base)][1] for p in range(P)])).to(DEV)
    ctx = Context(0)
    eps, C, m, st = ctx.nao_gen_eig(H, S, precision=precision)
    torch.cuda.synchronize()
    assert int(st.abs().sum()) == 0 and bool((m == n).all())
    for p in sorted({0, 1, len(base) - 1, P // 2, P - 1}):
        if p >= P:
            continue
        h, s = base[p % len(base)]
        L = np.linalg.cholesky(s)
        X = np.linalg.inv(L).conj().T
        Hp = X.conj().T @ h @ X
        e_ref = np.linalg.eigvalsh((Hp + Hp.conj().T) / 2)
        e, c = eps[p].cpu().numpy(), C[p].cpu().numpy()
        assert np.abs(e - e_ref).max() <= TOL_EPS * np.abs(e_ref).max()
        if precision == 0:
            res = np.linalg.norm(h @ c - s @ c * e[None, :]) / (n * np.linalg.norm(h, 2))
            assert res <= TOL_RES
            assert np.abs(c.conj().T @ s @ c - np.eye(n)).max() <= TOL_ORTH
    ctx.close()
