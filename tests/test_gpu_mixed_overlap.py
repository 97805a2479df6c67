"""Overlap of the mixed mode (GPU only): X from the Cholesky factor is FP64-accurate, as the
reduction of S is on the eigenvector route, up to the line ((tr S / n) tr S^-1 = 1e6) below which it
replaces that route.  With refinement 0 the vectors' C^H S C - 1 then comes from the 30- or 36-bit
products of H' and X V alone, where the eigenvector route adds its back-transformation of S: no
more than that route leaves, up to a factor of two for the largest of n^2 entries of each.  The
Rayleigh quotients meet the mixed mode's 1e-9 Ha bound at its default precision."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _pencils(n, P, cond, seed):
    """Overlaps with one weak direction that sets (tr S / n) tr S^-1 = cond, Hamiltonians with
    spectrum in [-1, 1] on the orthonormalised basis."""
    rng = np.random.Generator(np.random.PCG64(seed))

    def unitary():
        return np.linalg.qr(rng.normal(size=(n, n)) + 1j * rng.normal(size=(n, n)))[0]
    Hs, Ss = [], []
    for _ in range(P):
        s = 10.0 ** rng.uniform(-1.0, 0.0, n)
        s[0] = 0.0
        s *= n / s.sum()  # tr S / n = 1 up to the weak direction
        s[0] = 1.0 / (cond - (1.0 / s[1:]).sum())
        U, V = unitary(), unitary()
        S, Sh = (U * s) @ U.conj().T, (U * np.sqrt(s)) @ U.conj().T
        H = Sh @ (V * rng.uniform(-1.0, 1.0, n)) @ V.conj().T @ Sh
        Hs.append((H + H.conj().T) / 2)
        Ss.append((S + S.conj().T) / 2)
    return np.stack(Hs), np.stack(Ss)


@pytest.mark.parametrize("planes", [5, 6])
@pytest.mark.parametrize("n,cond", [(97, 9.5e5), (300, 3e5), (300, 9.5e5)])
def test_mixed_overlap_below_the_line(n, cond, planes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_4247_gb300.nao import NAO_MIXED_BF16X3, Context
    H, S = _pencils(n, 6, cond, 31 + n)
    Hd, Sd = torch.from_numpy(H).to(DEV), torch.from_numpy(S).to(DEV)
    fp64 = Context(0)
    ref = fp64.nao_gen_eig(Hd, Sd)[0].cpu().numpy()
    fp64.close()
    orth = {}
    for route, cfg in (("cholesky", {}), ("eigenvectors", {"overlap_mrrr": 0})):
        ctx = Context(0, config={"mixed_planes": planes, **cfg})
        ctx.nao_set_refinement(0)
        ctx.nao_profile_enable(True)
        eps, C, m, st = ctx.nao_gen_eig(Hd, Sd, precision=NAO_MIXED_BF16X3)
        torch.cuda.synchronize()
        assert ("overlap_chol" in ctx.nao_profile_read()) == (route == "cholesky")
        assert int(st.abs().sum()) == 0 and bool((m == n).all())
        C = C.cpu().numpy()
        orth[route] = np.abs(C.conj().transpose(0, 2, 1) @ S @ C - np.eye(n)).max()
        if planes == 6:
            assert np.abs(eps.cpu().numpy() - ref).max() <= 1e-9
        ctx.close()
    assert orth["cholesky"] <= 2.0 * orth["eigenvectors"], orth
