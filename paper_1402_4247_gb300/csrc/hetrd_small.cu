// Eigen_HH step 1 (Sec. 3, Procedures 1-6) for matrices that a cluster of blocks holds in shared
// memory: the whole reduction in one launch, FP64 arithmetic, unblocked.
//
// A small matrix is bound by the chain of short phases per column, not by arithmetic, so the
// design has as few of them as it can: one cluster barrier and three block barriers per column.
//  * Rows are dealt out in turn (row r to block r mod C), each block holding its rows in full
//    (columns 0 .. n-1 of the Hermitian matrix).
//  * The rank-2 update of a column is applied together with the next column's product, one pass
//    over the rows: A(r, c) -= v_r conj(w_c) + w_r conj(v_c) (the previous reflector's), then
//    q_r += A(r, c) x_c.
//  * The product runs on x, the unscaled column, while one warp forms the reflector from its
//    norm; p_r = (A v)_r = scale q_r + A(r, i+1) afterwards (v = (1, scale x)).
//  * Before the barrier a block pushes its p, its share of p^H v and, if it holds row i + 1, that
//    row into the shared memory of all blocks; after it every block forms w and the next column
//    x(r) = conj(A(i+1, r)) - tau p_r - v_r (conj(w_{i+1}) + a2) in full (a2 = -|tau|^2 p^H v / 2), so
//    there is no second exchange.  The exchange buffers alternate between two sets (a block can
//    be one column behind).
//  * An FP64 instruction holds its scheduler's pipe for 64 cycles, dependent or not, so scalars
//    are formed by one warp and reductions run only in warps that hold rows: with every warp
//    forming them redundantly a column took 15,000 cycles whatever n.
// FP64 work per column and block: 12 multiply-adds per element, 6 L^2 / C cycles (L trailing rows).
// Rule (hetrd_small_cluster): n^2 / C <= 6600, where that pass costs less than the panel's longer chain
// (csrc/hetrd.cu); up to n = 136, where the blocks are few (C = 1 up to n = 109, C = 2) and their exchange
// is short, 12000.  Whole reduction with digits and updates, this against panels, us:
//   C = 1, 150 problems: n = 64 569 / 924, 100 1605 / 1934, 109 1946 / 2034;
//   C = 2, 76 problems: n = 129 1785 / 2113, 136 2087 / 2281, 150 2752 / 2574;
//   C = 8, 10 problems: n = 100 718 / 1414, 200 2328 / 3046, 229 3113 / 3548;
//   C = 16, 1 to 7 problems: n = 64 423 / 792, 200 2094 / 2956, 305 4778 / 5102, 320 5300 / 5366.
// Clusters over nearly all SMs exchange more slowly and lose up to a tenth near the line: 9 problems
// (C = 16) n = 200 2761 / 3026, 256 4480 / 3914; 25 problems (C = 6) n = 140 1798 / 2042, 160 2443 / 2303.
#include <cooperative_groups.h>

#include "nao_internal.cuh"
#include "reflector.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int HS_THREADS = 256, HS_WARPS = HS_THREADS / 32;
constexpr int HS_ROWS = HS_THREADS - 32;  // threads that form vectors; the last warp forms scalars
constexpr int HS_MAX_CLUSTER = 16;
constexpr size_t HS_SMEM_LIMIT = 225 * 1024;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// store to the same shared-memory address of block k of the cluster
__device__ __forceinline__ void remote_store(const void* local, int k, double a) {
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"((uint32_t)__cvta_generic_to_shared(local)), "r"(k));
  asm volatile("st.shared::cluster.f64 [%0], %1;" :: "r"(ra), "d"(a) : "memory");
}

struct SmallSmem {
  int x, v, w, pb, rb, db, q, a;  // z64 units
  int Rld;                        // own rows, padded
  size_t bytes;
};

__host__ __device__ inline SmallSmem small_smem(int n, int C) {
  SmallSmem s;
  s.Rld = ((n + C - 1) / C + 7) / 8 * 8;
  int o = 0;
  s.x = o, o += n;
  s.v = o, o += n;
  s.w = o, o += n;
  s.pb = o, o += 2 * n;
  s.rb = o, o += 2 * n;
  s.db = o, o += 2 * HS_MAX_CLUSTER * HS_WARPS / 2;
  s.q = o, o += HS_WARPS * s.Rld;
  s.a = o, o += n * s.Rld;
  s.bytes = (size_t)o * sizeof(z64);
  return s;
}

__global__ void __launch_bounds__(HS_THREADS, 1)
hetrd_small_kernel(int n, const int32_t* __restrict__ size, z64* __restrict__ Abase, int ld, long long strideA,
                   double* __restrict__ dbase, double* __restrict__ ebase, z64* __restrict__ taubase, long long strideV) {
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  extern __shared__ z64 sm[];
  __shared__ z64 s_tau, s_scale, s_kappa;
  __shared__ double s_beta, s_a2, red[HS_WARPS];
  const int p = blockIdx.x / C;
  const int m = size ? size[p] : n;
  if (m <= 0) return;  // uniform over the cluster
  z64* A = Abase + (size_t)p * strideA;
  double* d = dbase + (size_t)p * strideV;
  double* e = ebase + (size_t)p * strideV;
  z64* tau = taubase + (size_t)p * strideV;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const SmallSmem L = small_smem(n, C);
  z64 *x = sm + L.x, *v = sm + L.v, *w = sm + L.w, *qp = sm + L.q, *As = sm + L.a;
  const int LW = (L.Rld + 31) >> 5;  // warps that hold own rows
  const int Rld = L.Rld, Rn = m > rank ? (m - rank + C - 1) / C : 0;  // own rows rank, rank + C, ...
  for (int idx = tid; idx < Rn * m; idx += HS_THREADS) {
    const int lr = idx % Rn, c = idx / Rn, r = lr * C + rank;
    z64 a = c <= r ? A[(size_t)c * ld + r] : zconj(A[(size_t)r * ld + c]);
    if (r == c) a.y = 0.0;
    As[(size_t)c * Rld + lr] = a;
  }
  double s = 0.0;
  if (wid < HS_WARPS - 1) {
    for (int r = tid; r < m; r += HS_ROWS) {
      const z64 a = A[r];
      x[r] = a;
      if (r > 1) s += zabs2(a);
    }
    s = warp_sum(s);
    if (lane == 0) red[wid] = s;
  }
  if (rank == 0 && tid == 0) d[0] = A[0].x;
  cluster.sync();  // (and every block's shared memory exists)

  for (int i = 0; i < m; ++i) {
    const int par = i & 1;
    if (i > 0) {
      // reflector i - 1: v, w and column i in full; x(i) is its diagonal element
      const z64 *pb = sm + L.pb + (par ^ 1) * n, *rb = sm + L.rb + (par ^ 1) * n;
      const z64 t = s_tau, scale = s_scale;
      const bool active = !(t.x == 0.0 && t.y == 0.0);
      if (wid == HS_WARPS - 1) {
        const double* db = (const double*)(sm + L.db) + (par ^ 1) * HS_MAX_CLUSTER * HS_WARPS;
        double dl = 0.0;  // p^H v
        for (int k = lane; k < C * LW; k += 32) dl += db[k];
        for (int o = 16; o > 0; o >>= 1)
          if (o < C * LW) dl += __shfl_xor_sync(0xffffffffu, dl, o);
        if (lane == 0) {
          const double a2 = active ? -0.5 * zabs2(t) * dl : 0.0;
          const z64 w0 = zmul(t, pb[i]);       // w_i = w0 + a2 (p = 0 when H = 1)
          s_a2 = a2;
          s_kappa = zmk(w0.x + 2.0 * a2, -w0.y);  // conj(w_i) + a2
        }
      } else {
        for (int r = i + tid; r < m; r += HS_ROWS) {
          z64 vr = zmk(0.0, 0.0), tp = zmk(0.0, 0.0);
          if (active) {
            vr = r == i ? zmk(1.0, 0.0) : zmul(x[r], scale);
            tp = zmul(t, pb[r]);
          }
          v[r] = vr;
          w[r] = tp;
        }
      }
      __syncthreads();
      if (i + 32 * wid < m && wid < HS_WARPS - 1) {
        const double a2 = s_a2;
        const z64 kappa = s_kappa;
        s = 0.0;
        for (int r = i + tid; r < m; r += HS_ROWS) {
          const z64 vr = v[r], tp = w[r];
          z64 xn = zfms(vr, kappa, zsub(zconj(rb[r]), tp));
          if (r == i) xn.y = 0.0;
          else if (r > i + 1) s = fma(xn.x, xn.x, fma(xn.y, xn.y, s));
          x[r] = xn;
          w[r] = zmk(fma(a2, vr.x, tp.x), fma(a2, vr.y, tp.y));
          if (r % C == rank) A[(size_t)(i - 1) * ld + r] = r == i ? zmk(s_beta, 0.0) : vr;  // Procedure 3
          if (r == i && rank == 0) d[i] = xn.x;
        }
        s = warp_sum(s);
        if (lane == 0) red[wid] = s;
      }
    }
    if (i == m - 1) {
      if (rank == 0 && tid == 0) {
        e[i] = 0.0;
        tau[i] = zmk(0.0, 0.0);
      }
      break;
    }
    __syncthreads();
    // Procedures 1-2 (the last warp) beside the pass over the own rows r > i: previous update and
    // product with x(i+2:).  Unit: eight rows, four lanes each, over a segment of the columns
    if (wid == HS_WARPS - 1) {
      const int nw = min(HS_WARPS - 1, (m - i + 31) >> 5);  // warps that left a part of the norm
      double n2 = red[0];
      if (nw > 1) {
        n2 = lane < nw ? red[lane] : 0.0;
#pragma unroll
        for (int o = HS_WARPS / 2; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
      }
      z64 t, scale;
      double beta;
      reflector(x[i + 1], n2, t, scale, beta);
      if (lane == 0) {
        s_tau = t;
        s_scale = scale;
        s_beta = beta;
        if (rank == 0) {
          e[i] = beta;
          tau[i] = t;
        }
      }
    }
    const int lr0 = i + 1 > rank ? (i + 1 - rank + C - 1) / C : 0, nl = max(Rn - lr0, 0);
    const int groups = (nl + 7) >> 3, cols = m - i - 1;
    // enough segments for six warps, of at least four columns per lane; the warps of the last one's
    // scheduler come last
    const int segs = groups > 0 ? max(1, min((HS_WARPS - 2 + groups - 1) / groups, cols >> 4)) : 1;
    const int wu = wid == 7 ? 7 : wid == 3 ? 6 : wid > 3 ? wid - 1 : wid;
    for (int u = wu; u < groups * segs; u += HS_WARPS) {
      const int lr = lr0 + 8 * (u / segs) + (lane & 7), sg = u % segs, r = lr * C + rank;
      const int c0 = i + 1 + sg * cols / segs, c1 = i + 1 + (sg + 1) * cols / segs;
      z64 q = zmk(0.0, 0.0);
      if (lr < Rn) {
        const z64 vr = i > 0 ? v[r] : zmk(0.0, 0.0), wr = i > 0 ? w[r] : zmk(0.0, 0.0);
        for (int c = c0 + (lane >> 3); c < c1; c += 4) {
          z64 a = As[(size_t)c * Rld + lr];
          if (i > 0) {
            a = zfmsc(wr, v[c], zfmsc(vr, w[c], a));
            if (c == r) a.y = 0.0;
            As[(size_t)c * Rld + lr] = a;
          }
          if (c > i + 1) q = zfma(a, x[c], q);
        }
      }
#pragma unroll
      for (int o = 8; o < 32; o <<= 1) {
        q.x += __shfl_xor_sync(0xffffffffu, q.x, o);
        q.y += __shfl_xor_sync(0xffffffffu, q.y, o);
      }
      if (lane < 8 && lr < Rn) qp[sg * Rld + lr] = q;
    }
    __syncthreads();
    // Procedure 4: p of the own rows, pushed to every block with the share of p^H v and row i + 1
    {
      const z64 t = s_tau, scale = s_scale;
      const bool active = !(t.x == 0.0 && t.y == 0.0);
      double dl = 0.0;
      for (int lr = lr0 + tid; lr < Rn; lr += HS_THREADS) {
        const int r = lr * C + rank;
        z64 pr = zmk(0.0, 0.0);
        if (active) {
          z64 q = qp[lr];
          for (int g = 1; g < segs; ++g) q = zadd(q, qp[g * Rld + lr]);
          pr = zfma(scale, q, As[(size_t)(i + 1) * Rld + lr]);
          const z64 vr = r == i + 1 ? zmk(1.0, 0.0) : zmul(x[r], scale);
          dl = fma(pr.x, vr.x, fma(pr.y, vr.y, dl));
        }
        const z64* o = sm + L.pb + par * n + r;
#pragma unroll 4
        for (int k = 0; k < C; ++k) {
          remote_store(&o->x, k, pr.x);
          remote_store(&o->y, k, pr.y);
        }
      }
      if (wid < LW) {
        if (32 * wid < nl) dl = warp_sum(dl);
        const double* od = (const double*)(sm + L.db) + par * HS_MAX_CLUSTER * HS_WARPS + rank * LW + wid;
        if (lane < C) remote_store(od, lane, dl);
      }
      if ((i + 1) % C == rank) {
        const int lr = (i + 1) / C;
        for (int c = i + 1 + tid; c < m; c += HS_THREADS) {
          const z64 a = As[(size_t)c * Rld + lr];
          const z64* o = sm + L.rb + par * n + c;
#pragma unroll 4
          for (int k = 0; k < C; ++k) {
            remote_store(&o->x, k, a.x);
            remote_store(&o->y, k, a.y);
          }
        }
      }
    }
    cluster.sync();
  }
}

void small_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int n, int nprob, int C, cudaStream_t st) {
  cfg.gridDim = dim3((unsigned)(nprob * C));
  cfg.blockDim = dim3(HS_THREADS);
  cfg.dynamicSmemBytes = small_smem(n, C).bytes;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
}

cudaError_t small_attributes() {
  cudaError_t e = cudaFuncSetAttribute(hetrd_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)HS_SMEM_LIMIT);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(hetrd_small_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

}  // namespace

// Blocks per matrix for the one-launch reduction (16, 8 .. 1; at most one per four rows, all clusters
// resident at once), or 0 where the blocked one is the faster.
int hetrd_small_cluster(int n, int nprob, int num_sms) {
  if (n > 640 || small_attributes() != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  for (int c = HS_MAX_CLUSTER; c > 0; c = c > 8 ? 8 : c - 1) {
    if (n * n > c * (n <= 136 ? 12000 : 6600)) return 0;
    if (c > 1 && (4 * c > n || (long long)nprob * c > num_sms)) continue;
    if (small_smem(n, c).bytes > HS_SMEM_LIMIT) return 0;
    if (c == 1) return 1;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    small_config(cfg, attr, n, nprob, c, nullptr);
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, hetrd_small_kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    if (clusters >= nprob) return c;
  }
  return 0;
}

cudaError_t launch_hetrd_small(int n, int nprob, const int32_t* size, z64* A, int ld, long long strideA, double* d, double* e,
                               z64* tau, long long strideV, int C, cudaStream_t st) {
  const cudaError_t err = small_attributes();
  if (err != cudaSuccess) return err;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  small_config(cfg, attr, n, nprob, C, st);
  return cudaLaunchKernelEx(&cfg, hetrd_small_kernel, n, size, A, ld, strideA, d, e, tau, strideV);
}
