"""Products with the Cholesky route's X over the range where X is not zero (GPU only): orders around
the products' tiles (128 rows, 16 or 32 columns, K steps of 16 with the second half of a complex
contraction 8 off), around a chunk of a long contraction, and in the two halves of a split
batch, against the pencil's own residuals."""
import numpy as np
import pytest

from paper_1402_4247_gb300 import synth
from tests.gpu_helpers import TOL_EPS, TOL_ORTH, TOL_RES

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n,problems,nb,split", [(16, 1, 16, 2), (127, 2, 40, 1), (128, 1, 128, 2), (129, 3, 129, 1), (136, 2, 1, 2),
                                                 (144, 2, 144, 2), (257, 5, 200, 1), (264, 1, 33, 2), (905, 2, 905, 2),
                                                 (1025, 1, 100, 2)])
def test_residuals(n, problems, nb, split):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_4247_gb300.nao import Context
    rng = np.random.Generator(np.random.PCG64(40 + n))
    H, S = synth.random_hermitian_pair(rng, n, cond=30.0)
    H = np.stack([H] + [H + np.diag(rng.uniform(-1, 1, n)) for _ in range(problems - 1)])
    Hd, Sd = torch.from_numpy(H).to(DEV), torch.from_numpy(S[None].copy()).to(DEV)
    smap = torch.zeros(problems, dtype=torch.int32, device=DEV)
    ctx = Context(0, config={"split_hprime": split})
    eps, C, m, st = ctx.nao_gen_eig(Hd, Sd, s_of_prob=smap, nb=nb)
    torch.cuda.synchronize()
    assert int(st.abs().sum()) == 0 and bool((m == n).all())
    for p in range(problems):
        c, e = C[p], eps[p, :nb].to(torch.complex128)
        hn = float(torch.linalg.matrix_norm(Hd[p], 2))
        assert float(torch.linalg.norm(Hd[p] @ c - Sd[0] @ c * e[None, :])) <= TOL_RES * n * hn
        assert float((c.conj().T @ Sd[0] @ c - torch.eye(nb, device=DEV)).abs().max()) <= TOL_ORTH
        if n <= 264:
            L = np.linalg.inv(np.linalg.cholesky(S))
            ref = np.linalg.eigvalsh(L @ H[p] @ L.conj().T)
            assert np.abs(eps[p].cpu().numpy() - ref).max() <= TOL_EPS * np.abs(ref).max()
    ctx.close()
