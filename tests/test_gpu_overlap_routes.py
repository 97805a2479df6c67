"""The two routes of the overlap (GPU only): X from the Cholesky factor where every direction is
kept and the overlap is well conditioned, from its eigendecomposition otherwise.  Batches that mix
both kinds (chosen per matrix on the device), padded orders, and orders at the edges of the
blocks, against the eigendecomposition alone (a setting of the context) and LAPACK."""
import numpy as np
import pytest

from paper_1402_4247_gb300 import synth
from tests.gpu_helpers import TOL_EPS, TOL_ORTH, TOL_RES

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _pencils(n, seed):
    """H, [S] of a well-conditioned overlap, one with an exact null direction (n > 2), one
    with an eigenvalue below the Cholesky route's bound but above the cut."""
    rng = np.random.Generator(np.random.PCG64(seed))
    H, S = synth.random_hermitian_pair(rng, n, cond=30.0)
    out = [S]
    if n > 2:
        S2 = S.copy()
        S2[:, 1] = S2[:, 0]
        S2[1, :] = S2[0, :]
        S2[1, 1] = S2[0, 0]
        out.append(S2)
        w, U = np.linalg.eigh(S)
        w[0] = 3e-9
        S3 = (U * w) @ U.conj().T
        out.append((S3 + S3.conj().T) / 2)
    return H, out


def _reference(H, S):
    s, U = np.linalg.eigh(S)
    X = U[:, s >= 1e-10] / np.sqrt(s[s >= 1e-10])
    Hp = X.conj().T @ H @ X
    return np.linalg.eigvalsh((Hp + Hp.conj().T) / 2), X.shape[1]


@pytest.mark.parametrize("n,copies", [(1, 3), (2, 1), (5, 1), (31, 1), (32, 1), (33, 40), (64, 1), (65, 1), (97, 2), (130, 1),
                                      (257, 60)])
def test_routes_agree(n, copies):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_4247_gb300.nao import Context
    H, Ss = _pencils(n, 700 + n)
    P = len(Ss) * copies
    Hd = torch.from_numpy(np.ascontiguousarray(H)).to(DEV).expand(P, n, n).contiguous()
    Sd = torch.from_numpy(np.stack(Ss)).to(DEV)
    smap = torch.arange(P, dtype=torch.int32, device=DEV) % len(Ss)
    # overlap_mrrr = 0 keeps every matrix on the eigendecomposition
    res = []
    for cfg in (None, {"overlap_mrrr": 0}):
        ctx = Context(0, config=cfg)
        eps, C, m, st = ctx.nao_gen_eig(Hd, Sd, s_of_prob=smap)
        torch.cuda.synchronize()
        assert int(st.abs().sum()) == 0
        res.append((eps.cpu().numpy(), C.cpu().numpy(), m.cpu().numpy()))
        ctx.close()
    for k, S in enumerate(Ss):
        e_ref, m_ref = _reference(H, S)
        hn = np.abs(e_ref).max()
        for p in (k, P - len(Ss) + k):
            (e, c, m), (e2, _, m2) = [(r[0][p], r[1][p], int(r[2][p])) for r in res]
            assert m == m2 == m_ref
            assert np.all(np.isinf(e[m:]))
            # FP64 routes of a pencil with s_min differ by ~eps |H'| |S| / s_min
            tol = TOL_EPS * hn if k < 2 else 1e-5 * hn
            assert np.abs(e[:m] - e_ref).max() <= tol and np.abs(e[:m] - e2[:m]).max() <= tol
            if k < 2:
                c = c[:, :m]
                # (a cut direction that H couples to leaves a residual in the full space)
                if m == n:
                    assert np.linalg.norm(H @ c - S @ c * e[None, :m]) <= TOL_RES * n * np.linalg.norm(H, 2)
                assert np.abs(c.conj().T @ S @ c - np.eye(m)).max() <= TOL_ORTH


def test_padded_orders_and_routes():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_4247_gb300.nao import Context
    n, orders = 70, (70, 33, 1, 64, 5)
    Hp = np.zeros((2 * len(orders), n, n), complex)
    Sp = np.zeros_like(Hp)
    ref = []
    for i, o in enumerate(orders):
        H, Ss = _pencils(o, 40 + o)
        for j in range(2):
            S = Ss[min(j, len(Ss) - 1)]
            Hp[2 * i + j, :o, :o] = H
            Sp[2 * i + j, :o, :o] = S
            ref.append((o,) + _reference(H, S))
    ctx = Context(0)
    size = torch.tensor([o for o in orders for _ in range(2)], dtype=torch.int32, device=DEV)
    eps, C, m, st = ctx.nao_gen_eig(torch.from_numpy(Hp).to(DEV), torch.from_numpy(Sp).to(DEV), s_size=size)
    torch.cuda.synchronize()
    assert int(st.abs().sum()) == 0
    eps, C, m = eps.cpu().numpy(), C.cpu().numpy(), m.cpu().numpy()
    ctx.close()
    for p, (o, e_ref, m_ref) in enumerate(ref):
        assert m[p] == m_ref
        assert np.abs(eps[p, :m_ref] - e_ref).max() <= TOL_EPS * np.abs(e_ref).max()
        assert np.all(np.isinf(eps[p, m_ref:])) and np.all(C[p][o:] == 0) and np.all(C[p][:, m_ref:] == 0)
        c = C[p][:o, :m_ref]
        assert np.abs(c.conj().T @ Sp[p][:o, :o] @ c - np.eye(m_ref)).max() <= TOL_ORTH
