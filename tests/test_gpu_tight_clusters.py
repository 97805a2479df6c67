"""Tight clusters of the tridiagonal solve (GPU only): overlaps with many exact null directions
(2 to 40 of them, one cluster each) and Hamiltonians whose spectrum has exactly and nearly
degenerate groups; kept count, eigenvalues and orthonormality against LAPACK."""
import numpy as np
import pytest

from tests.gpu_helpers import TOL_EPS, TOL_ORTH

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n,null,groups", [(40, 2, (3, 5)), (64, 12, (2, 2, 9)), (97, 33, (20, 4)), (150, 40, (37, 2, 3)), (120, 0, (60, 33, 2))])
def test_degenerate_groups(n, null, groups):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_4247_gb300.nao import Context
    rng = np.random.Generator(np.random.PCG64(n * 100 + null))

    def unitary(k):
        return np.linalg.qr(rng.normal(size=(k, k)) + 1j * rng.normal(size=(k, k)))[0]
    m = n - null
    s = np.concatenate([np.zeros(null), np.linspace(0.5, 2.0, m)])
    U = unitary(n)
    S = (U * s) @ U.conj().T
    S = (S + S.conj().T) / 2
    # H acts on the kept directions with the chosen spectrum: groups equal to 0, 1e-13 and 1e-12
    lam = np.sort(rng.uniform(-1.0, 1.0, m))
    k = 0
    for g, d in zip(groups, (0.0, 1e-13, 1e-12)):
        lam[k:k + g] = lam[k] + d * np.arange(g)
        k += g
    X = U[:, null:] * np.sqrt(s[null:])  # S = X X^H on the kept space
    V = unitary(m)
    H = X @ (V * lam) @ V.conj().T @ X.conj().T
    H = (H + H.conj().T) / 2
    ctx = Context(0)
    eps, C, mk, st = ctx.nao_gen_eig(torch.from_numpy(np.stack([H, H])).to(DEV), torch.from_numpy(np.stack([S, S])).to(DEV))
    torch.cuda.synchronize()
    assert int(st.abs().sum()) == 0
    ref = np.sort(lam)
    for p in range(2):
        assert int(mk[p]) == m
        e, c = eps[p, :m].cpu().numpy(), C[p, :, :m].cpu().numpy()
        assert np.abs(e - ref).max() <= TOL_EPS * max(1.0, np.abs(ref).max())
        assert np.abs(c.conj().T @ S @ c - np.eye(m)).max() <= TOL_ORTH
        # residual: H C = S C eps holds in the full space, H vanishes on the null directions
        assert np.linalg.norm(H @ c - S @ c * e[None, :]) <= 1e-12 * n * np.linalg.norm(H, 2)
    ctx.close()
