"""The Fermi-level kernel over its grid sizes (GPU only): from one value in one block to sets that
need every block, with ragged kept counts, gaps and nearly empty or full bands, against the
oracle's bisection."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n,nk,nspin,frac,kT", [
    (1, 1, 1, 0.5, 0.01), (3, 2, 2, 0.3, 0.02), (64, 4, 1, 0.25, 0.2), (512, 4, 1, 0.25, 0.01),
    (683, 3, 1, 0.999, 0.05), (700, 3, 2, 0.001, 0.05), (568, 64, 2, 0.25, 4e-4), (4096, 9, 2, 0.5, 0.01)])
def test_fermi_level_matches_oracle(n, nk, nspin, frac, kT):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_4247_gb300.nao import nao_fermi_level_noalloc
    rng = np.random.Generator(np.random.PCG64(n * 1000 + nk))
    P = nspin * nk
    eps = np.sort(rng.normal(0.0, 2.0, size=(P, n)), axis=1)
    m = rng.integers(max(1, n - n // 10), n + 1, size=P).astype(np.int32)
    for p in range(P):
        eps[p, m[p]:] = np.inf
    w = rng.uniform(0.5, 1.5, nk)
    w /= w.sum()
    g = 2.0 if nspin == 1 else 1.0
    ne = frac * g * sum(w[p % nk] * m[p] for p in range(P))
    mu_o, f_o, eb_o = oracle.fermi_occupations([eps[p, :m[p]] for p in range(P)], [w[p % nk] for p in range(P)], g, ne, kT)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
    f = torch.full((P, n), -1.0, dtype=torch.float64, device=DEV)
    mu, eb = (torch.empty(1, dtype=torch.float64, device=DEV) for _ in range(2))
    st = torch.full((1,), 7, dtype=torch.int32, device=DEV)
    nao_fermi_level_noalloc(t(w), t(eps), t(m), n, ne, kT, nspin, f, mu, eb, st)
    torch.cuda.synchronize()
    assert int(st[0]) == 0
    f = f.cpu().numpy()
    # N(mu) is a sum of at most P n terms of FP64 factors: its rounding, P n eps N_e at the worst
    count = g * sum(w[p % nk] * f[p, :m[p]].sum() for p in range(P))
    assert abs(count - ne) <= max(1e-13, P * n * 1.2e-16) * max(1.0, ne) * 4
    # occupations: df = f (1 - f) dmu / kT with dmu as the two counts allow
    for p in range(P):
        assert np.abs(f[p, :m[p]] - f_o[p]).max() <= 1e-9
        assert np.all(f[p, m[p]:] == 0.0)
    assert abs(float(eb[0]) - eb_o) <= 1e-9 * max(1.0, abs(eb_o))
