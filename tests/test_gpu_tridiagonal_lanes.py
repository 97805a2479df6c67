"""Eigenvalues of the tridiagonal solve over its lane counts (GPU only): the number of eigenvalues
decides how many lanes share one (16, 8, 4, 2, or one with a queue).  Spectra with clusters,
tiny and huge elements, split matrices (diagonal, block diagonal) and n = 1, against LAPACK."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _matrix(kind, n, rng):
    if kind == "random":
        A = rng.normal(size=(n, n)) + 1j * rng.normal(size=(n, n))
        return (A + A.conj().T) / 2
    if kind == "diagonal":
        return np.diag(rng.normal(size=n)).astype(complex)
    if kind == "blocks":  # two equal blocks: T splits, every eigenvalue twice
        k = max(1, n // 2)
        B = _matrix("random", k, rng)
        H = np.zeros((n, n), complex)
        H[:k, :k] = B
        H[k:2 * k, k:2 * k] = B
        return H
    w = np.concatenate([np.full(n - n // 3, 1.0), 1.0 + 1e-9 * np.arange(n // 3)]) if kind == "cluster" else np.logspace(-12, 6, n)
    Q = np.linalg.qr(rng.normal(size=(n, n)) + 1j * rng.normal(size=(n, n)))[0]
    H = (Q * w) @ Q.conj().T
    return (H + H.conj().T) / 2


@pytest.mark.parametrize("n,P", [(1, 5), (2, 1), (61, 19), (61, 30), (61, 70), (61, 150), (61, 200), (300, 4), (300, 33)])
@pytest.mark.parametrize("kind", ["random", "diagonal", "blocks", "cluster", "graded"])
def test_eigenvalues(n, P, kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_4247_gb300.nao import Context
    rng = np.random.Generator(np.random.PCG64(n * 1000 + P))
    base = [_matrix(kind, n, rng) for _ in range(3)]
    H = torch.from_numpy(np.stack([base[p % 3] for p in range(P)])).to(DEV)
    S = torch.eye(n, dtype=torch.complex128, device=DEV).expand(P, n, n).contiguous()
    ctx = Context(0)
    eps, _, m, st = ctx.nao_gen_eig(H, S, want_vectors=False)
    torch.cuda.synchronize()
    assert int(st.abs().sum()) == 0 and bool((m == n).all())
    e = eps.cpu().numpy()
    ctx.close()
    for p in sorted({0, min(1, P - 1), min(2, P - 1), P - 1}):
        ref = np.linalg.eigvalsh(base[p % 3])
        # bisection to a few eps |T|, reduction and LAPACK to n eps |H| each
        assert np.abs(e[p] - ref).max() <= 8 * n * 2.0 ** -52 * np.abs(ref).max()
