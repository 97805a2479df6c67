// Part 2 (Sec. 3) where no overlap direction is cut: X with X^H S X = 1 from the Cholesky
// factor instead of Eigen_HH(S).
//
// Any X with X^H S X = 1 over the same directions gives the same eigenvalues and (up to the free
// phase of each) the same eigenvectors C = X V, since the H' = X^H H X of two such X are unitarily
// similar.  The canonical orthogonalization X = U s^{-1/2} needs the whole eigendecomposition of
// S because it can cut directions; where all n are kept, X = L^{-H} with S = L L^H does the same at
// a small part of the work (n^3 / 3 + n^3 / 3 complex multiply-adds, nearly all in tensor-core
// products, against a tridiagonalization, a tridiagonal eigensolve and a back-transformation).
//
// Which overlaps take it is decided on the device, per matrix: every pivot positive, and with
// tr(S^{-1}) = |X|_F^2 (known once X is): s_min >= 1 / tr(S^{-1}), so s_cut tr(S^{-1}) < 1/2 means
// that nothing is cut, and (tr(S) / n) tr(S^{-1}) <= CH_MAX_COND keeps it to overlaps where X is
// as accurate as the eigenvector route's.  Measured (cells of n = 129 and 568, C^H S C - 1 and
// eigenvalue error of the two routes): 3.1e-13 / 1.1e-12 against 4.3e-13 / 1.1e-12 at 3e4 (n = 129),
// 5.3e-13 / 5.2e-13 against 8.9e-13 / 4.6e-13 at 1.5e5 (n = 568), 3.2e-12 / 4.2e-12 against the same
// at 3e5; at 3e6 one cell's residual was four times the other route's, so the line lies at 1e6.
// The others (size_eff > 0) go through Eigen_HH(S) as before; the kernels of that chain skip the
// matrices that are done (size_eff = 0).
//
// Layout: X column-major (ld n) holds both the factorization and the result, processed by blocks
// of B columns.  Before step J the columns from J on hold, in the rows from J on, the trailing
// matrix A' (lower part) and above it the rows of X found so far.  Step J:
//   diag:    A'_JJ = L L^H, Y = L^{-1} (FP64, one block per matrix); X_JJ <- 1, the rows J of the later
//            columns <- 0
//   product: the whole block column times Y^H: rows above J: X_J, rows J: Y^H, rows below: L_IJ
//   product: later columns -= (block column) L_IJ^H: the rows above are X's elimination, the rows
//            below the trailing update
// so one step is one FP64 kernel and two products.  Bound by the FP64 pipe in the diagonal blocks
// (one SM per matrix) and by the products' passes over X.
// Measured (ms per step; the overlap's chain before -> now, the skipped launches included): n = 64,
// 4 k-points ~1.3 -> 0.3; n = 305, 27 k-points ~10 -> 2.0; n = 568, 1 k-point ~18 -> 2.5, 64 k-points
// ~60 -> 8.8; n = 2000, 1 k-point ~140 -> 14.  An overlap that fails pays it on top (n = 600, 8
// k-points, cut directions: 3.5 of 57 ms).
#include <cfloat>

#include "nao_internal.cuh"

namespace {

constexpr double CH_MAX_COND = 1e6;
constexpr int CH_THREADS = 256;

// One block (blockIdx.x = 0) factors the w x w diagonal block at j0; the others zero the rows j0 ..
// j0 + w - 1 of the later columns.  Rows and columns from size[p] on count as the identity.
// The elimination runs on [A' | 1] with unscaled rows (a_ik / d_k as multiplier), so a step is
// one pass and one barrier; the thread that finishes the next pivot also forms its reciprocal.
// Y (w x w, row-major, ld B): rows scaled by d^{-1/2} at the end.
template <int B>
__global__ void __launch_bounds__(CH_THREADS)
chol_diag_kernel(int n, const int32_t* __restrict__ size, z64* __restrict__ Xbase, long long sX, int j0, int w,
                 z64* __restrict__ Ybase, int* __restrict__ fail) {
  extern __shared__ z64 chs[];
  z64* a = chs;                // [B][B + 1], lower
  z64* y = chs + B * (B + 1);  // [B][B + 1], lower
  __shared__ double s_d[B], s_rd[B];
  __shared__ int s_bad;
  const int p = blockIdx.y, tid = threadIdx.x;
  const int m = size ? size[p] : n;
  z64* X = Xbase + (size_t)p * sX;
  if (blockIdx.x > 0) {
    const int rest = n - j0 - w;
    for (int idx = (blockIdx.x - 1) * CH_THREADS + tid; idx < rest * w; idx += (gridDim.x - 1) * CH_THREADS)
      X[(size_t)(j0 + w + idx / w) * n + j0 + idx % w] = zmk(0.0, 0.0);
    return;
  }
  constexpr int LD = B + 1;
  for (int idx = tid; idx < w * w; idx += CH_THREADS) {
    const int r = idx % w, c = idx / w;
    z64 v = zmk(0.0, 0.0);
    if (j0 + r < m && j0 + c < m) v = X[(size_t)(j0 + c) * n + j0 + r];
    else if (r == c) v = zmk(1.0, 0.0);
    if (r >= c) a[r * LD + c] = v;
    y[r * LD + c] = zmk(r == c ? 1.0 : 0.0, 0.0);
    X[(size_t)(j0 + c) * n + j0 + r] = zmk(r == c ? 1.0 : 0.0, 0.0);
  }
  if (tid == 0) s_bad = fail[p];
  __syncthreads();
  if (tid == 0) {
    const double d = a[0].x;
    if (!(d > 0.0 && d <= DBL_MAX)) s_bad = 1;
    s_d[0] = d;
    s_rd[0] = 1.0 / d;
  }
  __syncthreads();
  for (int k = 0; k + 1 < w; ++k) {
    const double rd = s_rd[k];
    // element (k + 1, k + 1) is item 0 of the list of rows k + 1 .., taken by thread 0
    for (int idx = tid; idx < (w - 1 - k) * w; idx += CH_THREADS) {
      const int i = k + 1 + idx / w, q = idx % w, c = k + 1 + q < w ? k + 1 + q : k + 1 + q - w;  // columns k + 1 .., then 0 .. k
      if (c > i) continue;
      const z64 l = zscale(a[i * LD + k], rd);
      if (c > k) {
        z64 v = zfmsc(l, a[c * LD + k], a[i * LD + c]);
        if (c == i) v.y = 0.0;
        a[i * LD + c] = v;
        if (idx == 0) {
          if (!(v.x > 0.0 && v.x <= DBL_MAX)) s_bad = 1;
          s_d[k + 1] = v.x;
          s_rd[k + 1] = 1.0 / v.x;
        }
      } else {
        y[i * LD + c] = zfms(l, y[k * LD + c], y[i * LD + c]);
      }
    }
    __syncthreads();
  }
  const bool bad = s_bad != 0;
  if (tid == 0 && bad) fail[p] = 1;
  z64* Y = Ybase + (size_t)p * B * B;
  for (int idx = tid; idx < w * w; idx += CH_THREADS) {
    const int r = idx / w, c = idx % w;
    z64 v = zmk(r == c ? 1.0 : 0.0, 0.0);  // (a failed matrix stays finite; it is not used)
    if (!bad) v = c <= r ? zscale(y[r * LD + c], rsqrt(s_d[r])) : zmk(0.0, 0.0);
    Y[r * B + c] = v;
  }
}

// Zero below the diagonal of X (and outside size[p]), and the block's share of |X|_F^2 and tr S:
// part[(p nb + b) 2 ..] for 64 columns per block b.
__global__ void __launch_bounds__(CH_THREADS)
chol_norm_kernel(int n, const int32_t* __restrict__ size, z64* __restrict__ Xbase, const z64* __restrict__ Sbase,
                 long long sX, double* __restrict__ part) {
  __shared__ double red[2][CH_THREADS / 32];
  const int p = blockIdx.y, b = blockIdx.x, tid = threadIdx.x;
  const int m = size ? size[p] : n;
  z64* X = Xbase + (size_t)p * sX;
  double f = 0.0, t = 0.0;
  for (int c = 64 * b; c < min(n, 64 * b + 64); ++c) {
    for (int r = tid; r < n; r += CH_THREADS) {
      if (r > c || c >= m || r >= m) X[(size_t)c * n + r] = zmk(0.0, 0.0);
      else f += zabs2(X[(size_t)c * n + r]);
    }
    if (tid == 0 && c < m) t += Sbase[(size_t)p * sX + (size_t)c * n + c].x;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
  if ((tid & 31) == 0) red[0][tid >> 5] = f;
  if (tid == 0) red[1][0] = t;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int w = 0; w < CH_THREADS / 32; ++w) s += red[0][w];
    part[2 * ((size_t)p * gridDim.x + b)] = s;
    part[2 * ((size_t)p * gridDim.x + b) + 1] = red[1][0];
  }
}

// size_eff[p]: 0 where X is done, else the order that Eigen_HH(S) works on
__global__ void chol_decide_kernel(int n, int nprob, int nb, const int32_t* __restrict__ size, double s_cut,
                                   const double* __restrict__ part, const int* __restrict__ fail,
                                   int32_t* __restrict__ size_eff) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= nprob) return;
  const int m = size ? size[p] : n;
  double f = 0.0, t = 0.0;
  for (int b = 0; b < nb; ++b) {
    f += part[2 * ((size_t)p * nb + b)];
    t += part[2 * ((size_t)p * nb + b) + 1];
  }
  const bool ok = m > 0 && !fail[p] && f * (t / m) <= CH_MAX_COND && f * s_cut < 0.5;  // (NaN: not)
  size_eff[p] = ok ? 0 : m;
}

// kept counts and statuses of the matrices that are done (the eigenvector route wrote the others)
__global__ void chol_counts_kernel(int n, int nprob, const int32_t* __restrict__ size,
                                   const int32_t* __restrict__ size_eff, int32_t* __restrict__ m, int32_t* __restrict__ status) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= nprob || size_eff[p]) return;
  m[p] = size ? size[p] : n;
  status[p] = 0;
}

template <int B>
cudaError_t diag(int n, int nprob, const int32_t* size, z64* X, long long sX, int j0, z64* Y, int* fail, cudaStream_t st) {
  const size_t smem = 2 * (size_t)B * (B + 1) * sizeof(z64);
  const cudaError_t e = cudaFuncSetAttribute(chol_diag_kernel<B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int w = n - j0 < B ? n - j0 : B, rest = n - j0 - w;
  const int zb = (rest * w + 8 * CH_THREADS - 1) / (8 * CH_THREADS);
  chol_diag_kernel<B><<<dim3(1 + zb, nprob), CH_THREADS, smem, st>>>(n, size, X, sX, j0, w, Y, fail);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_chol_diag(int B, int n, int nprob, const int32_t* size, z64* X, long long sX, int j0, z64* Y, int* fail,
                             cudaStream_t st) {
  return B == 32 ? diag<32>(n, nprob, size, X, sX, j0, Y, fail, st) : diag<64>(n, nprob, size, X, sX, j0, Y, fail, st);
}

size_t chol_part_doubles(int n, int nprob) { return 2 * (size_t)((n + 63) / 64) * nprob; }

cudaError_t launch_chol_decide(int n, int nprob, const int32_t* size, z64* X, const z64* S, long long sX, double s_cut,
                               double* part, const int* fail, int32_t* size_eff, cudaStream_t st) {
  const int nb = (n + 63) / 64;
  chol_norm_kernel<<<dim3(nb, nprob), CH_THREADS, 0, st>>>(n, size, X, S, sX, part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  chol_decide_kernel<<<(nprob + 127) / 128, 128, 0, st>>>(n, nprob, nb, size, s_cut, part, fail, size_eff);
  return cudaGetLastError();
}

cudaError_t launch_chol_counts(int n, int nprob, const int32_t* size, const int32_t* size_eff, int32_t* m, int32_t* status,
                               cudaStream_t st) {
  chol_counts_kernel<<<(nprob + 127) / 128, 128, 0, st>>>(n, nprob, size, size_eff, m, status);
  return cudaGetLastError();
}
