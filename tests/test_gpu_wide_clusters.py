"""Clusters of more than 32 eigenvalues that are together wider than the tight band (1e-11 |T|)
(GPU only): members a band apart are not taken out of one another, overlap by up to 1e-5 and are
left to the Newton-Schulz steps, each of which squares the overlaps; the second of them brings
1e-10 to rounding: C^H C - 1 of n eigenvectors below 1e-14."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n,P,group,delta", [(120, 20, 40, 1e-12), (120, 20, 33, 9e-12), (200, 6, 100, 5e-12)])
def test_wide_clusters_end_orthonormal(n, P, group, delta):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_4247_gb300.nao import Context
    rng = np.random.Generator(np.random.PCG64(n + group))
    lam = np.sort(rng.uniform(-1.0, 1.0, (P, n)), axis=1)
    for i in range(0, n - group + 1, group):
        lam[:, i:i + group] = lam[:, i:i + 1] + delta * np.arange(group)
    V = np.linalg.qr(rng.normal(size=(P, n, n)) + 1j * rng.normal(size=(P, n, n)))[0]
    H = (V * lam[:, None, :]) @ V.conj().transpose(0, 2, 1)
    H = (H + H.conj().transpose(0, 2, 1)) / 2
    S = np.broadcast_to(np.eye(n, dtype=complex), H.shape).copy()
    ctx = Context(0)
    eps, C, m, st = ctx.nao_gen_eig(torch.from_numpy(H).to(DEV), torch.from_numpy(S).to(DEV))
    torch.cuda.synchronize()
    ctx.close()
    assert int(st.abs().sum()) == 0 and bool((m == n).all())
    C = C.cpu().numpy()
    assert np.abs(C.conj().transpose(0, 2, 1) @ C - np.eye(n)).max() <= 1e-14
    res = np.linalg.norm(H @ C - C * eps.cpu().numpy()[:, None, :], axis=1).max()
    assert res <= 1e-12 * n
