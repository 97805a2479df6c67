"""Residuals of the eigenvectors of tight clusters (GPU only), over many matrices: a member may carry
the rounding of its solve over the share of its norm that the others leave (at least a half, else
it is solved for again), twice that of an isolated eigenvector, and as much again from the
members that were taken out of it.  So the largest |H c - eps c| over groups of equal and
nearly equal eigenvalues stays within three times the largest of the same spectra without groups.
Groups that span more than the tight band (25 eigenvalues 1e-12 apart) end orthonormal too."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("delta", [0.0, 1e-14, 1e-12])
@pytest.mark.parametrize("n,P,group", [(12, 600, 2), (24, 200, 4), (48, 100, 12), (100, 40, 25)])
def test_groups_against_separate_eigenvalues(n, P, group, delta):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_4247_gb300.nao import Context
    ctx = Context(0)
    worst = []
    for grouped in (False, True):
        rng = np.random.Generator(np.random.PCG64(n + group))
        lam = np.sort(rng.uniform(-1.0, 1.0, (P, n)), axis=1)
        if grouped:
            for i in range(0, n - group + 1, group):
                lam[:, i:i + group] = lam[:, i:i + 1] + delta * np.arange(group)
        V = np.linalg.qr(rng.normal(size=(P, n, n)) + 1j * rng.normal(size=(P, n, n)))[0]
        H = (V * lam[:, None, :]) @ V.conj().transpose(0, 2, 1)
        H = (H + H.conj().transpose(0, 2, 1)) / 2
        S = np.broadcast_to(np.eye(n, dtype=complex), H.shape).copy()
        eps, C, m, st = ctx.nao_gen_eig(torch.from_numpy(H).to(DEV), torch.from_numpy(S).to(DEV))
        torch.cuda.synchronize()
        assert int(st.abs().sum()) == 0 and bool((m == n).all())
        C = C.cpu().numpy()
        worst.append(np.linalg.norm(H @ C - C * eps.cpu().numpy()[:, None, :], axis=1).max())
        assert np.abs(C.conj().transpose(0, 2, 1) @ C - np.eye(n)).max() <= 1e-14
    ctx.close()
    assert worst[1] <= 3.0 * worst[0], worst
