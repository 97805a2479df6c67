// Part 5 (Sec. 3): chemical potential and band energy.  mu solves
//   N(mu) = g sum_p w_p sum_{j < m_p} f((eps_pj - mu)/kT) = N_e,  f(x) = 1/(1 + e^x),
// by safeguarded Newton steps on [min eps - 40 kT, max eps + 40 kT] (N is strictly increasing
// for kT > 0), then f_pj and E_band = g sum w f eps.  All eigenvalues of all (k, spin) problems
// enter one sum, so the kernel runs on the whole GPU: each round every block sums its share of
// the Fermi factors and of their derivatives, the partial sums meet after a grid-wide barrier,
// and every block takes the same (deterministic, fixed-order) step.
//
// What bounds it is the chain of rounds: FP64 arithmetic at 64 cycles per warp instruction and
// scheduler (an exponential and a division per value, ~45 instructions), reductions, and a grid
// barrier of ~1.2 us.  Hence:
//  * Newton steps, with bisection where a step leaves the bracket or the bracket does not
//    halve, and the bracket closed around the root at the end: ~15-30 rounds instead of the
//    ~55 of plain bisection;
//  * f is evaluated only within FP_WIN kT of mu (1 below, 0 above: e^-60 is 1e-10 of the last
//    bit of a sum that holds any occupied state), so the early rounds are comparisons;
//  * the blocks' partial sums are added by one warp (in every thread they cost 152 FP64
//    instructions per warp and round, ~10 us);
//  * small sets take few blocks (one: no grid barrier) and few warps (a reduction per warp).
// Measured on GB300: 72,704 eigenvalues 1713 -> 500 us, 256 eigenvalues 1393 -> 200 us.
#include <cooperative_groups.h>

#include <cfloat>

#include "nao_internal.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int FT = 256;

__device__ __forceinline__ double fermi_fn(double x) {
  if (x <= 0.0) return 1.0 / (1.0 + exp(x));
  const double ex = exp(-x);
  return ex / (1.0 + ex);
}

__device__ double block_minmax(double v, double* red, bool is_max) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double u = __shfl_xor_sync(0xffffffffu, v, o);
    v = is_max ? fmax(v, u) : fmin(v, u);
  }
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double t = red[0];
  for (int k = 1; k < (int)(blockDim.x >> 5); ++k) t = is_max ? fmax(t, red[k]) : fmin(t, red[k]);
  return t;
}

constexpr int FP_SUMS = 3;         // sums per round: states below mu, their and the others' tails, dN/dmu
constexpr double FP_WIN = 60.0;    // f is 1 below and 0 above this many kT from mu

// Grid-wide sums of v[0..K) in a fixed order, into out[0..K) of every thread; buf alternates so
// that a fast block never overwrites partials that a slow block is still reading.
// red: 8 K doubles of shared memory at least, tot: K.  active (uniform over a warp): false for a
// warp whose values are all zero.
template <int K>
__device__ void grid_sum(cg::grid_group& grid, const double* v, double* out, double* red, double* tot, double* scratch,
                         int& buf, bool active) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double x[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    x[k] = v[k];
    if (active)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x[k] += __shfl_xor_sync(0xffffffffu, x[k], o);
  }
  __syncthreads();
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) red[wid * K + k] = x[k];
  __syncthreads();
  double* part = scratch + (size_t)buf * FP_SUMS * gridDim.x;
  buf ^= 1;
  if (threadIdx.x < K) {
    double t = 0.0;
    for (int w = 0; w < FT / 32; ++w) t += red[w * K + threadIdx.x];
    if (gridDim.x == 1) tot[threadIdx.x] = t;
    else part[(size_t)blockIdx.x * K + threadIdx.x] = t;
  }
  if (gridDim.x > 1) {
    grid.sync();
    if (wid == 0) {
      double t[K];
#pragma unroll
      for (int k = 0; k < K; ++k) t[k] = 0.0;
      for (unsigned b = lane; b < gridDim.x; b += 32)
#pragma unroll
        for (int k = 0; k < K; ++k) t[k] += __ldcg(part + (size_t)b * K + k);
#pragma unroll
      for (int k = 0; k < K; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t[k] += __shfl_xor_sync(0xffffffffu, t[k], o);
        if (lane == 0) tot[k] = t[k];
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) out[k] = tot[k];
}

__global__ void __launch_bounds__(FT)
fermi_kernel(int n, int nprob, int nk, double g, const double* __restrict__ wk, const double* __restrict__ eps,
             const int32_t* __restrict__ m, int nb, double n_electrons, double kT, double f_min,
             double* __restrict__ f, int32_t* __restrict__ nocc, double* __restrict__ mu_out, double* __restrict__ eband_out,
             int32_t* __restrict__ status, double* __restrict__ scratch) {
  cg::grid_group grid = cg::this_grid();
  __shared__ double red[8 * FP_SUMS > 32 ? 8 * FP_SUMS : 32], tot[FP_SUMS], mmx[2];
  __shared__ int s_over;
  int buf = 0;
  const size_t total = (size_t)nprob * n;
  const size_t gtid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  // threads that take values: at least two each, in whole groups of four warps (one per scheduler)
  const size_t gall = (size_t)gridDim.x * blockDim.x, gwant = ((total + 1) / 2 + 127) / 128 * 128;
  const size_t gstride = gwant < gall ? gwant : gall;
  const bool busy = gtid < gstride;

  double lmin = DBL_MAX, lmax = -DBL_MAX, cap = 0.0;
  for (size_t idx = busy ? gtid : total; idx < total; idx += gstride) {
    const int p = (int)(idx / n), j = (int)(idx % n);
    if (j < m[p]) {
      const double e = eps[idx];
      lmin = fmin(lmin, e);
      lmax = fmax(lmax, e);
      cap += g * wk[p % nk];
    }
    if (j == 0) nocc[p] = 0;
  }
  // min and max through the sum machinery: two grid sums of +-large sentinels would lose
  // precision, so reduce them with dedicated partial slots
  lmin = block_minmax(lmin, red, false);
  lmax = block_minmax(lmax, red, true);
  double* mm = scratch + 2 * FP_SUMS * (size_t)gridDim.x;
  if (threadIdx.x == 0) {
    mm[2 * blockIdx.x] = lmin;
    mm[2 * blockIdx.x + 1] = lmax;
  }
  grid_sum<1>(grid, &cap, &cap, red, tot, scratch, buf, busy);  // (contains a grid.sync)
  double emin = lmin, emax = lmax;
  if (gridDim.x > 1) {
    if (threadIdx.x < 32) {
      for (unsigned b = threadIdx.x; b < gridDim.x; b += 32) {
        emin = fmin(emin, __ldcg(mm + 2 * b));
        emax = fmax(emax, __ldcg(mm + 2 * b + 1));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        emin = fmin(emin, __shfl_xor_sync(0xffffffffu, emin, o));
        emax = fmax(emax, __shfl_xor_sync(0xffffffffu, emax, o));
      }
      if (threadIdx.x == 0) {
        mmx[0] = emin;
        mmx[1] = emax;
      }
    }
    __syncthreads();
    emin = mmx[0];
    emax = mmx[1];
  }
  int32_t st = 0;
  if (!(n_electrons >= 0.0 && n_electrons <= cap * (1.0 + 1e-14)) || !(emin <= emax)) st = NAO_E_RANGE;
  double lo = emin - 40.0 * kT, hi = emax + 40.0 * kT, root = DBL_MAX;
  if (st == 0) {
    const double rkT = 1.0 / kT;
    double x = 0.5 * (lo + hi), width2 = hi - lo;  // bracket width two rounds ago
    double width1 = width2, reach = 1.0;
    for (int it = 0; it < 200; ++it) {
      const double mid = 0.5 * (lo + hi), tol = 1e-15 * fmax(1.0, fabs(mid));
      if (mid <= lo || mid >= hi || hi - lo <= tol) break;
      // N - N_e = (states below x - N_e) + tails, the tails (f above x, f - 1 below) summed by
      // themselves: inside a gap N is flat to its rounding, and only their sum places mu
      double s[FP_SUMS] = {0.0, 0.0, 0.0};
      for (size_t idx = busy ? gtid : total; idx < total; idx += gstride) {
        const int p = (int)(idx / n), j = (int)(idx % n);
        if (j >= m[p]) continue;
        const double t = (eps[idx] - x) * rkT, w = wk[p % nk];
        if (!(t > 0.0)) s[0] += w;
        if (!(fabs(t) > FP_WIN)) {
          const double ex = exp(-fabs(t)), r = 1.0 / (1.0 + ex);
          const double q = ex * r;  // min(f, 1 - f)
          s[1] = fma(t > 0.0 ? w : -w, q, s[1]);
          s[2] = fma(w, q * r, s[2]);  // f (1 - f) = kT df/dmu
        }
      }
      grid_sum<FP_SUMS>(grid, s, s, red, tot, scratch, buf, busy);
      const double excess = fma(g, s[0], -n_electrons) + g * s[1];
      const bool below = excess < 0.0;
      if (below) lo = x;
      else hi = x;
      const double step = -excess * kT / (g * s[2]);
      double xn = x + step;
      root = xn;
      if (!(fabs(step) > 16.0 * tol)) {  // at the root: close the bracket from its other side
        const double w = fmax(2.0 * fabs(step), tol) * reach;
        xn = below ? x + w : x - w;
        reach *= 8.0;
      } else if (hi - lo > 0.5 * width2) {  // Newton while the bracket halves every two rounds
        xn = hi;                            // (bisects)
      }
      width2 = width1;
      width1 = hi - lo;
      x = (xn > lo && xn < hi) ? xn : 0.5 * (lo + hi);
    }
  }
  // The last Newton point: the bracket's ends are iterates, one of them next to the root, so its middle
  // would be half of the last width off (mean |mu - root| / 1e-15 max(1, |mu|) 0.36, bisection 0.16)
  const double mu = (root >= lo && root <= hi) ? root : 0.5 * (lo + hi);
  // occupations, band energy, occupied-band counts
  double eb = 0.0;
  for (size_t idx = busy ? gtid : total; idx < total; idx += gstride) {
    const int p = (int)(idx / n), j = (int)(idx % n);
    double fj = 0.0;
    if (st == 0 && j < m[p]) {
      fj = fermi_fn((eps[idx] - mu) / kT);
      eb += g * wk[p % nk] * fj * eps[idx];
      if (fj > f_min) atomicMax(&nocc[p], j + 1);
    }
    f[idx] = fj;
  }
  grid_sum<1>(grid, &eb, &eb, red, tot, scratch, buf, busy);  // (its barriers publish nocc)
  if (blockIdx.x == 0) {
    if (threadIdx.x == 0) {
      *mu_out = (st == 0) ? mu : __longlong_as_double(0x7ff8000000000000ll);
      *eband_out = (st == 0) ? eb : __longlong_as_double(0x7ff8000000000000ll);
      s_over = 0;
    }
    __syncthreads();
    // bands beyond the nb returned eigenvectors must be empty; the count is clamped so
    // that the density-matrix product never reads past column nb
    for (int p = threadIdx.x; p < nprob; p += blockDim.x)
      if (__ldcg(nocc + p) > nb) {
        s_over = 1;
        nocc[p] = nb;
      }
    __syncthreads();
    if (threadIdx.x == 0 && status) *status = (st == 0 && s_over) ? (int32_t)NAO_E_INVALID : st;
  }
}

}  // namespace

size_t fermi_scratch_doubles(int num_sms) { return (size_t)(2 * FP_SUMS + 2) * num_sms + 64; }

cudaError_t launch_fermi(int num_sms, int n, int nprob, int nk, double g, const double* wk, const double* eps,
                         const int32_t* m, int nb, double n_electrons, double kT, double f_min, double* f,
                         int32_t* nocc, double* mu, double* eband, int32_t* status, double* scratch, cudaStream_t st) {
  int per_sm = 0;
  cudaError_t err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fermi_kernel, FT, 0);
  if (err != cudaSuccess) return err;
  if (per_sm < 1) return cudaErrorCooperativeLaunchTooLarge;
  // eight values per thread before another block joins (its share of a round's barrier costs
  // more than eight comparisons), at most one block per SM
  const long long want = ((long long)n * nprob + 8 * FT - 1) / (8 * FT);
  int grid = want < num_sms ? (int)want : num_sms;
  void* args[] = {&n,  &nprob, &nk,   &g,  &wk,    &eps,   &m,       &nb,     &n_electrons,
                  &kT, &f_min, &f,    &nocc, &mu,  &eband, &status, &scratch};
  return cudaLaunchCooperativeKernel((const void*)fermi_kernel, dim3(grid), dim3(FT), args, 0, st);
}

// ---------------------------------------------------------------------------------------
// Allocation-free variant of Part 5 (no counterpart in the paper).
//
// The entry point above takes its scratch (grid partial sums, per-problem occupied-band
// counts) from the context's workspace, which the library grows with cudaMalloc.  Some
// callers cannot allow that: host codes that hand the library a fixed device-memory pool
// and forbid allocations behind their back (DFT drivers in Fortran/MPI with their own
// allocators), and serving loops that must never synchronise the device in the middle
// of a step (cudaMalloc/cudaFree can synchronise).  For them nao_fermi_level_noalloc
// runs the same kernel on a scratch array that is part of the library image itself.
// ---------------------------------------------------------------------------------------

#include <mutex>

namespace {
constexpr int NOALLOC_MAX_BLOCKS = 512;            // grid blocks whose partial sums fit
constexpr int NOALLOC_MAX_PROBLEMS = 65536;        // (spin, k) problems whose band counts fit
constexpr size_t NOALLOC_PART_DOUBLES = 8 * (size_t)NOALLOC_MAX_BLOCKS + 64;
static_assert(2 * FP_SUMS + 2 <= 8, "the grid's partial sums fit");
constexpr size_t NOALLOC_DOUBLES = NOALLOC_PART_DOUBLES + NOALLOC_MAX_PROBLEMS / 2;  // + int32 counts
}  // namespace

// 288.5 KiB (295,424 bytes) of device memory, held by every GPU that loads the library until
// the process exits.
static __device__ __align__(256) double nao_fermi_scratch[NOALLOC_DOUBLES];

namespace {
std::mutex g_noalloc_mu;
constexpr int NOALLOC_MAX_DEVICES = 64;
void* g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};

// Device address of nao_fermi_scratch on the current device, looked up once per device and
// kept for the life of the process (a cudaDeviceReset of the device in between would leave
// it stale; the entry point's documentation excludes that).  In host code the symbol names
// a host-side shadow, not device memory.
cudaError_t noalloc_scratch(int dev, double** out) {
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return cudaErrorInvalidDevice;
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, nao_fermi_scratch);
    if (e != cudaSuccess) return e;
    g_noalloc_ptr[dev] = p;
  }
  *out = (double*)g_noalloc_ptr[dev];
  return cudaSuccess;
}
}  // namespace

extern "C" int nao_fermi_level_noalloc(int n, int nspin, int nk, const double* wk, const double* eps,
                                       const int32_t* m_kept, int nb, double n_electrons, double kT, double* f_out,
                                       double* mu_out, double* eband_out, int32_t* status, void* stream) {
  if (n < 1 || nk < 1 || (nspin != 1 && nspin != 2) || nb < 1 || nb > n)
    return nao_fail(nullptr, NAO_E_INVALID, "nao_fermi_level_noalloc: bad sizes");
  if ((long long)nspin * nk > NOALLOC_MAX_PROBLEMS)
    return nao_fail(nullptr, NAO_E_INVALID,
                    "nao_fermi_level_noalloc: %d problems exceed the fixed scratch limit of %d",
                    nspin * nk, NOALLOC_MAX_PROBLEMS);
  if (!wk || !eps || !m_kept || !f_out || !mu_out || !eband_out || !status)
    return nao_fail(nullptr, NAO_E_INVALID, "nao_fermi_level_noalloc: NULL array");
  if (!(kT > 0.0)) return nao_fail(nullptr, NAO_E_INVALID, "nao_fermi_level_noalloc: kT must be > 0");
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  double* scratch = nullptr;
  if (e == cudaSuccess) e = noalloc_scratch(dev, &scratch);
  if (e != cudaSuccess)
    return nao_fail(nullptr, NAO_E_CUDA, "nao_fermi_level_noalloc: %s", cudaGetErrorString(e));
  const int grid = sms < NOALLOC_MAX_BLOCKS ? sms : NOALLOC_MAX_BLOCKS;
  int32_t* nocc = (int32_t*)(scratch + NOALLOC_PART_DOUBLES);
  e = launch_fermi(grid, n, nspin * nk, nk, nspin == 1 ? 2.0 : 1.0, wk, eps, m_kept, nb, n_electrons, kT,
                   NAO_F_MIN_DEFAULT, f_out, nocc, mu_out, eband_out, status, scratch, (cudaStream_t)stream);
  if (e != cudaSuccess)
    return nao_fail(nullptr, NAO_E_CUDA, "nao_fermi_level_noalloc: launch failed: %s", cudaGetErrorString(e));
  return NAO_OK;
}
