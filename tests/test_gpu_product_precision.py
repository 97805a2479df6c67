"""Precision of the tensor-core products at FP64 accuracy (GPU only): operands are held to 63 bits below
their row's (column's) power of two, and of the digit products only those below 2^-71 of the two
scales are dropped, whatever the length of the contraction.

* All digits at their largest, of one sign, in every plane: rows whose entries lie below the row's
  scale by 2^0 to 2^-40 (the entry that sets the scale meets a zero), at the longest chunk, against
  the exact integers.  Bound: the dropped products, at most 12 pairs of |d d'| <= 2^8 at 2^-71, 11
  at 2^-76 .. (12.4 2^-63 per term), and one rounding of the result.
* Random graded operands, large entries of A meeting small ones of B: the root mean square error
  against extended precision is that of the dropped products, digits uniform over 32 values
  (variance 85.25) in 12 pairs of 2 K terms: 85.25 sqrt(24 K) 2^-71 of the scales, allowed twice."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_4247_gb300.nao import Context
    c = Context(0)
    yield c
    c.close()


def _product(ctx, A, B):
    from paper_1402_4247_gb300.nao import NAO_GEMM_TC
    C = ctx.nao_zgemm(torch.from_numpy(A[None]).to(DEV), torch.from_numpy(B[None]).to(DEV), method=NAO_GEMM_TC)
    torch.cuda.synchronize()
    return C.cpu().numpy()[0]


@pytest.mark.parametrize("K", [257, 1232, 1233])
@pytest.mark.parametrize("ga,gb", [(0, 0), (0, 40), (40, 0), (20, 20), (5, 35), (30, 15)])
@pytest.mark.parametrize("digit", [-16, 15])
def test_largest_digits(ctx, K, ga, gb, digit):
    M, N = 3, 2
    # digit planes 1 .. 11 (or 1 .. 10, 53 bits) of the 63-bit integer, moved down by g bits
    ndig = 11 if digit < 0 else 10
    pat = sum(digit * 32 ** (11 - j) for j in range(ndig))

    def entry(g):
        v = abs(pat) >> g
        top = max(0, v.bit_length() - 53)  # what a double holds
        return (v >> top << top) * (-1 if digit < 0 else 1)
    a, b = entry(ga), entry(gb)
    A = np.full((M, K), float(a), dtype=complex) * (1 + 1j)
    B = np.full((K, N), float(b), dtype=complex) * (1 + 1j)
    big = float(2 ** 62)  # sets a scale of 2^63, meets a zero
    A[:, 0], B[0, :] = big, 0.0
    A[:, 1], B[1, :] = 0.0, big
    got = _product(ctx, A, B)
    exact = 2 * a * b * (K - 2)  # imaginary part; the real part cancels
    tol = 2 * K * 12.4 * 2.0 ** 63 + abs(exact) * 2.0 ** -52
    for z in got.ravel():
        assert abs(int(z.imag) - exact) <= tol
        assert abs(int(z.real)) <= 2 * K * 12.4 * 2.0 ** 63


@pytest.mark.parametrize("K", [100, 177, 256, 257, 300, 1232, 1500, 2500])
def test_graded_operands(ctx, K):
    rng = np.random.Generator(np.random.PCG64(K))
    M, N = 40, 36
    g = rng.integers(0, 21, K)
    A = (rng.normal(size=(M, K)) + 1j * rng.normal(size=(M, K))) * 2.0 ** -g
    B = (rng.normal(size=(K, N)) + 1j * rng.normal(size=(K, N))) * (2.0 ** (g - 20.0))[:, None]
    err = _product(ctx, A, B) - A.astype(np.clongdouble) @ B.astype(np.clongdouble)
    scale = lambda X, ax: 2.0 ** (1 + np.floor(np.log2(np.maximum(np.abs(X.real), np.abs(X.imag)).max(ax))))  # noqa: E731
    rel = err / (scale(A, 1)[:, None] * scale(B, 0)[None, :])
    rms = float(np.sqrt((rel.real ** 2 + rel.imag ** 2).mean() / 2))
    assert rms <= 2 * 85.25 * np.sqrt(24 * K) * 2.0 ** -71
