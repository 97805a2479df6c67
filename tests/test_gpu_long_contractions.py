"""Tensor-core products of more than 176 terms (352 real), formed from e4m3 digits (GPU only): operands
of 20-bit integers, whose digits beyond the fifth are zero and whose products and sums are exact
in FP64, must come back exactly.  Orders around the tiles (128 rows, 16 columns), the K steps of 32
with both halves of a complex contraction, the chunks of 1344, and the largest digit sums."""
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


@pytest.mark.parametrize("largest", [False, True], ids=["random", "largest"])
@pytest.mark.parametrize("P,M,N,K,tA,tB", [
    (1, 33, 18, 176, 0, 0), (2, 131, 17, 177, 2, 1), (1, 1, 1, 257, 0, 0), (2, 127, 15, 264, 0, 1), (3, 128, 16, 272, 2, 0), (1, 129, 17, 273, 1, 2), (2, 31, 33, 288, 0, 2),
    (1, 300, 100, 289, 2, 2), (1, 16, 257, 1343, 0, 0), (1, 130, 40, 1344, 2, 1), (1, 65, 31, 1345, 1, 0), (1, 20, 18, 2700, 0, 2)])
def test_integer_products(ctx, P, M, N, K, tA, tB, largest):
    from paper_1402_4247_gb300.nao import NAO_GEMM_TC
    rng = np.random.Generator(np.random.PCG64(M + 10 * N + 100 * K))

    def operand(r, c):
        top = 2 ** 19 - 1
        re, im = (rng.integers(-top, top + 1, size=(P, r, c)) for _ in range(2))
        if largest:  # every product of one sign in the real or the imaginary part
            re, im = np.full_like(re, top), np.full_like(im, top)
        return torch.from_numpy(re + 1j * im).to(DEV)

    A = operand(K, M) if tA else operand(M, K)
    B = operand(N, K) if tB else operand(K, N)
    op = lambda X, t: X if t == 0 else (X.transpose(1, 2) if t == 1 else X.transpose(1, 2).conj())  # noqa: E731
    got = ctx.nao_zgemm(A, B, transA=tA, transB=tB, method=NAO_GEMM_TC)
    torch.cuda.synchronize()
    a, b = op(A, tA), op(B, tB)
    ar, ai, br, bi = a.real.contiguous(), a.imag.contiguous(), b.real.contiguous(), b.imag.contiguous()
    assert torch.equal(got.real, ar @ br - ai @ bi) and torch.equal(got.imag, ar @ bi + ai @ br)
