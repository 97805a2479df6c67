"""Orders at the edges of the back-transformation's blocks (one block of 64 reflectors, one of 128,
their halves partly or wholly empty, several blocks), against the oracle (GPU only)."""
import numpy as np
import pytest

import oracle
from paper_1402_4247_gb300 import synth
from tests.gpu_helpers import check_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n", [2, 17, 33, 64, 65, 66, 81, 129, 130, 194])
def test_eigenvectors_at_block_edges(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_4247_gb300.nao import Context
    rng = np.random.Generator(np.random.PCG64(500 + n))
    pairs = [synth.random_hermitian_pair(rng, n, cond=50.0) for _ in range(3)]
    H = torch.from_numpy(np.stack([h for h, _ in pairs])).to(DEV)
    S = torch.from_numpy(np.stack([s for _, s in pairs])).to(DEV)
    ctx = Context(0)
    eps, C, m, st = ctx.nao_gen_eig(H, S)
    torch.cuda.synchronize()
    eps, C, m, st = (t.cpu().numpy() for t in (eps, C, m, st))
    ctx.close()
    for p, (h, s) in enumerate(pairs):
        assert st[p] == 0
        e_o, C_o, m_o = oracle.generalized_eigensolve(h, s)[:3]
        check_problem(h, s, eps[p], C[p], int(m[p]), e_o, C_o, m_o, label=f"n={n} p={p}")
