// Eigen_HH steps 3-4 (Sec. 3: "rearrangement of eigenvectors" and "normalization") and the
// small element-wise steps around them.  The eigenvectors of A are U = Q Z with
// Q = H_0 H_1 ... H_{m-2} from the tridiagonalization; Q is applied in compact WY blocks
// (Q_j = I - V_j T_j V_j^H: W = V_j^H U, then U -= (V_j T_j) W, products issued by the caller), then
// the columns are scaled to unit 2-norm.  For the overlap matrix the normalization also
// applies Part 2's canonical orthogonalization X = U_m diag(s_m^{-1/2}).
#include "nao_internal.cuh"

namespace {

__device__ __forceinline__ double wsum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__global__ void count_kept_kernel(int n, int nprob, const int32_t* __restrict__ size, const double* __restrict__ w,
                                  long long strideV, double s_cut, int32_t* __restrict__ m,
                                  int32_t* __restrict__ status) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= nprob) return;
  const double* wp = w + (size_t)p * strideV;
  const int np = size ? size[p] : n;  // the problem's order: eigenvalues 0 .. np-1
  int k = 0;
  for (int j = 0; j < np; ++j) k += (wp[j] >= s_cut);
  m[p] = k;
  if (k == 0 && status[p] == 0) status[p] = NAO_E_ALLCUT;
}

__global__ void hermitize_kernel(int n, const int32_t* __restrict__ size, z64* __restrict__ Abase, int ld,
                                 long long strideA) {
  const int p = blockIdx.z;
  const int m = size ? size[p] : n;
  const int r = blockIdx.x * blockDim.x + threadIdx.x;  // row
  const int c = blockIdx.y;                             // column
  if (r >= m || c >= m || r > c) return;
  z64* A = Abase + (size_t)p * strideA;
  if (r == c) {
    A[(size_t)c * ld + r].y = 0.0;
  } else {
    A[(size_t)c * ld + r] = zconj(A[(size_t)r * ld + c]);  // upper (r < c) from lower (c, r)
  }
}

__global__ void write_eps_kernel(int n, int nprob, const int32_t* __restrict__ m, const double* __restrict__ w,
                                 long long strideV, double* __restrict__ eps) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)n * nprob) return;
  const int p = (int)(idx / n), j = (int)(idx % n);
  eps[idx] = (j < m[p]) ? w[(size_t)p * strideV + j] : __longlong_as_double(0x7ff0000000000000ll);
}

__global__ void zero_cols_kernel(int n, int nprob, int nb, const int32_t* __restrict__ m, z64* __restrict__ C) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)n * nb * nprob) return;
  const int p = (int)(idx / ((size_t)n * nb));
  const int j = (int)(idx % nb);
  if (j >= m[p]) C[idx] = zmk(0.0, 0.0);
}

__global__ void scale_cols_sqrt_kernel(int n, int nprob, int nb, const z64* __restrict__ C, const double* __restrict__ f,
                                       z64* __restrict__ Cs) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)n * nb * nprob) return;
  const int p = (int)(idx / ((size_t)n * nb));
  const int j = (int)(idx % nb);
  const double fj = f[(size_t)p * n + j];
  Cs[idx] = zscale(C[idx], fj > 0.0 ? sqrt(fj) : 0.0);
}

// Ce = Cs diag(eps) over the occupied columns (eps is +inf where f = 0: those stay zero)
__global__ void scale_cols_eps_kernel(int n, int nprob, int nb, const z64* __restrict__ Cs, const double* __restrict__ f,
                                      const double* __restrict__ eps, z64* __restrict__ Ce) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)n * nb * nprob) return;
  const int p = (int)(idx / ((size_t)n * nb));
  const int j = (int)(idx % nb);
  const double fj = f[(size_t)p * n + j];
  Ce[idx] = fj > 0.0 ? zscale(Cs[idx], eps[(size_t)p * n + j]) : zmk(0.0, 0.0);
}

}  // namespace

cudaError_t launch_count_kept(int n, int nprob, const int32_t* size, const double* w, long long strideV, double s_cut,
                              int32_t* m, int32_t* status, cudaStream_t st) {
  count_kept_kernel<<<(nprob + 127) / 128, 128, 0, st>>>(n, nprob, size, w, strideV, s_cut, m, status);
  return cudaGetLastError();
}

cudaError_t launch_hermitize(int n, int nprob, const int32_t* size, z64* A, int ld, long long strideA, cudaStream_t st) {
  dim3 grid((n + 127) / 128, n, nprob);
  hermitize_kernel<<<grid, 128, 0, st>>>(n, size, A, ld, strideA);
  return cudaGetLastError();
}

cudaError_t launch_write_eps(int n, int nprob, const int32_t* m, const double* w, long long strideV, double* eps,
                             cudaStream_t st) {
  const size_t tot = (size_t)n * nprob;
  write_eps_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(n, nprob, m, w, strideV, eps);
  return cudaGetLastError();
}

cudaError_t launch_zero_cols(int n, int nprob, int nb, const int32_t* m, z64* C, cudaStream_t st) {
  const size_t tot = (size_t)n * nb * nprob;
  zero_cols_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(n, nprob, nb, m, C);
  return cudaGetLastError();
}

cudaError_t launch_scale_cols_eps(int n, int nprob, int nb, const z64* Cs, const double* f, const double* eps, z64* Ce,
                                  cudaStream_t st) {
  const size_t tot = (size_t)n * nb * nprob;
  scale_cols_eps_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(n, nprob, nb, Cs, f, eps, Ce);
  return cudaGetLastError();
}

cudaError_t launch_scale_cols_sqrt(int n, int nprob, int nb, const z64* C, const double* f, z64* Cs, cudaStream_t st) {
  const size_t tot = (size_t)n * nb * nprob;
  scale_cols_sqrt_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(n, nprob, nb, C, f, Cs);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Blocked form of steps 3-4 (compact WY): Q = Q_0 Q_1 ... with Q_j = H_{j nb} ... H_{j nb+nb-1}
// = I - V_j T_j V_j^H, applied as two matrix products per block with V_j T_j formed once (run
// on the tensor cores by the caller).  The kernels below prepare the operands.
// ---------------------------------------------------------------------------------------
namespace {

// Vfull(:, i) = explicit reflector i (1 at row i + off, A(r, i) below, 0 elsewhere) for
// i < m - off, zero columns otherwise (ncolv >= n columns); tauc[i] = tau[i] or 0.
__global__ void extract_v_kernel(int n, const int32_t* __restrict__ size, const z64* __restrict__ Abase, int lda,
                                 long long strideA, const z64* __restrict__ taubase, long long strideV, int ncolv,
                                 z64* __restrict__ Vbase, int ldv, long long strideVf, z64* __restrict__ taucbase,
                                 int off) {
  const int p = blockIdx.z;
  const int m = size ? size[p] : n;
  const int i = blockIdx.y;  // column
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n || i >= ncolv || m == 0) return;  // (order 0: nothing reads the result)
  const z64* A = Abase + (size_t)p * strideA;
  z64 val = zmk(0.0, 0.0);
  if (i < m - off) {
    if (r == i + off) val = zmk(1.0, 0.0);
    else if (r > i + off && r < m) val = A[(size_t)i * lda + r];
  }
  Vbase[(size_t)p * strideVf + (size_t)i * ldv + r] = val;
  if (r == 0) taucbase[(size_t)p * ncolv + i] = (i < m - off) ? taubase[(size_t)p * strideV + i] : zmk(0.0, 0.0);
}

// U(:, c) = Z(:, m - nc + c) (or Z(:, c) when lowest) as complex for c < nc, rows < m; zero
// elsewhere (n x n).
__global__ void init_u_kernel(int n, const int32_t* __restrict__ size, const int32_t* __restrict__ ncols,
                              const double* __restrict__ Zbase, int ldz, long long strideZ, z64* __restrict__ Ubase,
                              int ldu, long long strideU, int lowest) {
  const int p = blockIdx.z;
  const int m = size ? size[p] : n;
  const int nc = ncols ? ncols[p] : m;
  const int c = blockIdx.y;
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n || m == 0) return;  // (order 0: U is left alone)
  double v = 0.0;
  if (c < nc && r < m) v = Zbase[(size_t)p * strideZ + (size_t)(lowest ? c : m - nc + c) * ldz + r];
  Ubase[(size_t)p * strideU + (size_t)c * ldu + r] = zmk(v, 0.0);
}

// T (nb x nb, row-major, upper triangular) of block j from G = V^H V (row-major, Hermitian):
// T_ii = tau_i, T(0:i, i) = -tau_i T(0:i, 0:i) G(0:i, i).  One block of 256 threads forms the
// diagonal BT_H x BT_H part of T (of sub-block blockIdx.x % nsub) in shared memory, by halves:
//   T = [T11 T12; 0 T22] with T12 = -T11 (G12 T22),
// from 16 x 16 diagonal blocks formed by the column recurrence (a warp each, two lanes per
// row) through 16 -> 32 -> 64; the caller joins the two halves of a 128-column block with
// two tensor-core products.  FP64 bounds it (64^3/6 complex multiply-adds, 40 us of one SM's
// FP64 pipe, with every lane busy; one thread per row over the whole block, the form before, was a
// chain of 128^2/2 multiply-adds).  Back-transformation stage per step, before -> now: n = 64, 4
// problems 2.82 -> 0.49 ms; n = 129, 12 problems 2.87 -> 0.77 ms; n = 568, 128 problems 39.8 -> 36.8 ms.
// G and T of block j of problem p at (j nprob + p) nb^2.
constexpr int BT_H = NAO_WY_T;
constexpr int BT_THREADS = 256;
constexpr int BT_LD = BT_H + 1;

// X = G12 T22, then T12 = -T11 X for the pairs of h x h blocks along the diagonal
template <int H>
__device__ __forceinline__ void bt_join(const z64* __restrict__ g, z64* __restrict__ t, z64* __restrict__ x) {
  constexpr int NP = BT_H / (2 * H), TOT = NP * H * H;
  static_assert(TOT % BT_THREADS == 0, "whole passes");
#pragma unroll
  for (int o = 0; o < TOT / BT_THREADS; ++o) {  // lanes along the rows: one c (and k range) per warp
    const int idx = threadIdx.x + o * BT_THREADS;
    const int pr = idx / (H * H), r = idx % H, c = (idx / H) % H, b = pr * 2 * H;
    z64 acc = zmk(0.0, 0.0);
    for (int k = 0; k <= c; ++k) acc = zfma(g[(b + r) * BT_LD + b + H + k], t[(b + H + k) * BT_LD + b + H + c], acc);
    x[(pr * H + r) * (H + 1) + c] = acc;
  }
  __syncthreads();
#pragma unroll
  for (int o = 0; o < TOT / BT_THREADS; ++o) {  // lanes along the columns: one r (and k range) per warp
    const int idx = threadIdx.x + o * BT_THREADS;
    const int pr = idx / (H * H), c = idx % H, r = (idx / H) % H, b = pr * 2 * H;
    z64 acc = zmk(0.0, 0.0);
    for (int k = r; k < H; ++k) acc = zfma(t[(b + r) * BT_LD + b + k], x[(pr * H + k) * (H + 1) + c], acc);
    t[(b + r) * BT_LD + b + H + c] = zmk(-acc.x, -acc.y);
  }
  __syncthreads();
}

__global__ void __launch_bounds__(BT_THREADS)
build_t_kernel(int nb, int nprob, int nsub, const z64* __restrict__ Gbase, const z64* __restrict__ taucbase,
               int ncolv, z64* __restrict__ Tbase) {
  extern __shared__ z64 bts[];
  z64* g = bts;                       // [BT_H][BT_LD]
  z64* t = g + BT_H * BT_LD;          // [BT_H][BT_LD]
  z64* x = t + BT_H * BT_LD;          // [BT_H / 2][BT_H / 2 + 1]
  const int q = blockIdx.x / nsub, p = q % nprob, j = q / nprob;
  const int s0 = blockIdx.x % nsub * BT_H, H = nb - s0 < BT_H ? nb - s0 : BT_H;  // this sub-block's columns
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const z64* G = Gbase + (size_t)q * nb * nb + (size_t)s0 * nb + s0;
  const z64* tau = taucbase + (size_t)p * ncolv + (size_t)j * nb + s0;
  z64* T = Tbase + (size_t)q * nb * nb;
  // rows s0 .. of T outside the diagonal sub-block: zero (the join writes the upper ones)
  for (int idx = tid; idx < H * nb; idx += BT_THREADS) {
    const int r = idx / nb, c = idx % nb;
    if (c < s0 || c >= s0 + H) T[(size_t)(s0 + r) * nb + c] = zmk(0.0, 0.0);
  }
  bool any = false;
  if (tid < H) any = tau[tid].x != 0.0 || tau[tid].y != 0.0;
  if (!__syncthreads_or(any)) {  // no reflector here: T = 0
    for (int idx = tid; idx < H * H; idx += BT_THREADS)
      T[(size_t)(s0 + idx / H) * nb + s0 + idx % H] = zmk(0.0, 0.0);
    return;
  }
  for (int idx = tid; idx < BT_H * BT_H; idx += BT_THREADS) {
    const int r = idx / BT_H, c = idx % BT_H;
    g[r * BT_LD + c] = (r < H && c < H) ? G[(size_t)r * nb + c] : zmk(0.0, 0.0);
    t[r * BT_LD + c] = zmk(0.0, 0.0);
  }
  __syncthreads();
  if (wid < BT_H / 16) {  // T(r, i) = -tau_i sum_{r <= c < i} T(r, c) G(c, i) on the diagonal blocks
    const int b = 16 * wid, r = lane & 15, h = lane >> 4;
    for (int i = 0; i < 16; ++i) {
      const z64 ti = b + i < H ? tau[b + i] : zmk(0.0, 0.0);
      z64 acc = zmk(0.0, 0.0);
      for (int c = h; c < i; c += 2) acc = zfma(t[(b + r) * BT_LD + b + c], g[(b + c) * BT_LD + b + i], acc);
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 16);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 16);
      if (h == 0 && r <= i) t[(b + r) * BT_LD + b + i] = r == i ? ti : zmul(zmk(-ti.x, -ti.y), acc);
      __syncwarp();
    }
  }
  __syncthreads();
  bt_join<16>(g, t, x);
  if (BT_H > 32) bt_join<32>(g, t, x);
  for (int idx = tid; idx < H * H; idx += BT_THREADS) {
    const int r = idx / H, c = idx % H;
    T[(size_t)(s0 + r) * nb + s0 + c] = t[r * BT_LD + c];
  }
}

// column c < nc: U(:, c) /= ||U(:, c)||, times 1/sqrt(w[m - nc + c]) when use_rsqrt
__global__ void normalize_cols_kernel(int n, const int32_t* __restrict__ size, const int32_t* __restrict__ ncols,
                                      const double* __restrict__ wbase, long long strideV, int use_rsqrt,
                                      z64* __restrict__ Ubase, int ldu, long long strideU) {
  const int p = blockIdx.y;
  const int m = size ? size[p] : n;
  const int nc = ncols ? ncols[p] : m;
  const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (c >= nc) return;
  z64* u = Ubase + (size_t)p * strideU + (size_t)c * ldu;
  double s = 0.0;
  for (int r = lane; r < m; r += 32) s += zabs2(u[r]);
  s = wsum(s);
  double sc = 1.0 / sqrt(s);
  if (use_rsqrt) sc /= sqrt(wbase[(size_t)p * strideV + (m - nc + c)]);
  for (int r = lane; r < m; r += 32) u[r] = zscale(u[r], sc);
}

}  // namespace

cudaError_t launch_extract_v(int n, int nprob, const int32_t* size, const z64* A, int lda, long long strideA,
                             const z64* tau, long long strideV, int ncolv, z64* V, int ldv, long long strideVf,
                             z64* tauc, int off, cudaStream_t st) {
  dim3 grid((n + 127) / 128, ncolv, nprob);
  extract_v_kernel<<<grid, 128, 0, st>>>(n, size, A, lda, strideA, tau, strideV, ncolv, V, ldv, strideVf, tauc, off);
  return cudaGetLastError();
}

cudaError_t launch_init_u(int n, int nprob, const int32_t* size, const int32_t* ncols, const double* Z, int ldz,
                          long long strideZ, z64* U, int ldu, long long strideU, int lowest, cudaStream_t st) {
  dim3 grid((n + 127) / 128, n, nprob);
  init_u_kernel<<<grid, 128, 0, st>>>(n, size, ncols, Z, ldz, strideZ, U, ldu, strideU, lowest);
  return cudaGetLastError();
}

cudaError_t launch_build_t(int nb, int nprob, int nblk, const z64* G, const z64* tauc, int ncolv, z64* T,
                           cudaStream_t st) {
  const size_t smem = (2 * (size_t)BT_H * BT_LD + (size_t)(BT_H / 2) * (BT_H / 2 + 1)) * sizeof(z64);
  const cudaError_t e = cudaFuncSetAttribute(build_t_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int nsub = (nb + BT_H - 1) / BT_H;
  build_t_kernel<<<nprob * nblk * nsub, BT_THREADS, smem, st>>>(nb, nprob, nsub, G, tauc, ncolv, T);
  return cudaGetLastError();
}

cudaError_t launch_normalize_cols(int n, int nprob, const int32_t* size, const int32_t* ncols, const double* w,
                                  long long strideV, int use_rsqrt, z64* U, int ldu, long long strideU,
                                  cudaStream_t st) {
  dim3 grid((n + 7) / 8, nprob);
  normalize_cols_kernel<<<grid, 256, 0, st>>>(n, size, ncols, w, strideV, use_rsqrt, U, ldu, strideU);
  return cudaGetLastError();
}
