"""Precision of the Fermi level at small smearing (GPU only), where f(1 - f) / kT times an error of mu
is what N and the occupations lose.  The kernel's bracket closes to 1e-15 max(1, |mu|); bisection
leaves mu uniformly inside a bracket between half of that and all of it, a mean error of at most a
quarter.  So the mean over many sets of |mu - root| (root in extended precision) may be no more
than 0.25e-15 max(1, |mu|)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_mean_error_of_mu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_4247_gb300.nao import nao_fermi_level_noalloc
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
    errors = []
    for seed in range(160):
        rng = np.random.Generator(np.random.PCG64(seed))
        nspin, nk, n = int(rng.integers(1, 3)), int(rng.integers(1, 9)), int(10.0 ** rng.uniform(0.0, 2.5))
        P, kT, g = nspin * nk, 10.0 ** rng.uniform(-4.5, -2.5), 2.0 if nspin == 1 else 1.0
        eps = np.sort(rng.normal(size=(P, n)) * 10.0 ** rng.uniform(-1.0, 1.0), axis=1)
        w = rng.uniform(0.1, 1.0, nk)
        w /= w.sum()
        # an electron count that some level shares: its own occupation at a level's energy
        wl = np.tile(w, nspin).astype(np.longdouble)[:, None]
        target = np.longdouble(eps.ravel()[int(rng.integers(P * n))]) + kT * rng.uniform(-2.0, 2.0)

        def count(x):
            z = np.clip((eps.astype(np.longdouble) - x) / np.longdouble(kT), -11000, 11000)
            return g * (wl / (1 + np.exp(z))).sum()
        ne = float(count(target))
        lo, hi = target - 1e-6, target + 1e-6  # the root for the rounded ne
        for _ in range(70):
            x = (lo + hi) / 2
            lo, hi = (x, hi) if count(x) < ne else (lo, x)
        f = torch.empty((P, n), dtype=torch.float64, device=DEV)
        mu, eb = (torch.empty(1, dtype=torch.float64, device=DEV) for _ in range(2))
        st = torch.empty(1, dtype=torch.int32, device=DEV)
        m = np.full(P, n, dtype=np.int32)
        nao_fermi_level_noalloc(t(w), t(eps), t(m), n, ne, kT, nspin, f, mu, eb, st)
        torch.cuda.synchronize()
        assert int(st[0]) == 0
        errors.append(float(abs(np.longdouble(float(mu[0])) - x)) / (1e-15 * max(1.0, abs(float(x)))))
    assert np.mean(errors) <= 0.25, np.mean(errors)
