// Eigen_HH step 1 (Sec. 3, Procedures 1-6) with exact digit products on the tensor cores: one
// panel of NAO_HT_NB columns of the blocked Householder reduction (see csrc/hetrd_fp64.cu for the
// notation and the FP64 form).
//
// The Hermitian product p = A22 v of every column (Procedure 4) is formed from 8-bit digits: once per panel every
// row r of the trailing matrix (both triangles) is scaled by its own power of two 2^{e_r}
// (|a| < 2^{e_r}) and q = round(a 2^{8S-2-e_r}) written in S balanced base-256 digits (S = 8:
// 62 bits, FP64 accuracy with margin for entries below their row maximum; S = 6: 46 bits, the
// H' reduction of the mixed mode); per column v (|v| <= 1) is split the same way.  The digit
// products run on mma.sync m16n8k16 with f16 operands (integers up to 2^11 are exact) and FP32
// accumulators: the A operand holds 16 rows of one digit plane s, the B operand all eight digit
// planes t of v side by side (its eight columns), so one instruction forms the products of
// plane s with every plane of v.  |d d'| <= 2^14 and two products per column, so 512 columns
// stay below 2^24 and every FP32 sum is an exact integer; the sums are then combined as
// sum_{s,t} R_st 2^{-8 (s + t)} in integer arithmetic (orders beyond s + t = 7 + 3 dropped).
//   Rates per SM (measured): f16 mma.sync 1019 MAC per clock, the integer dot product DP4A 252
// (mma.sync on 8-bit integers runs at that rate too).  A digit is converted from its byte by
// one byte permute per two digits into 1024 + u and one packed subtraction.
//
// The panel was bound by the serial part of each column (27 us at n = 64, 46 us at n = 568
// on four SMs): FP64 reduction trees, division chains, four barriers.  Here
//  * a column takes two cluster barriers (block barriers when one block holds the matrix): one
//    after the product, one after the next column has been formed.  The dot product of
//    Procedure 5 needs no third: p^H v = p_raw^H v - 2 Re(y1^H y2) with y1 = W^H v, y2 = V^H v;
//  * up to 16 blocks share a matrix (tiles of 16 rows dealt out in turn), each keeping its own
//    rows of the panel's V and W in shared memory where they fit; where a column and its digits (48 n
//    bytes) do not, the column lies in the digits' space, for one more barrier and pass over v a
//    column (digits to n = 3649);
//  * a block pushes its rows of the next column straight into the shared memory of the
//    others, so that after the barrier the column is local everywhere;
//  * the panel's own products (V^H v and W^H v, the corrections V y1 + W y2, the next column's
//    updates) run on the same digit MMAs, in eight warps beside the eight that form A22 v: in
//    FP64 they took as long as the product (an FP64 warp instruction holds its scheduler's
//    pipe for 64 cycles, and every reduction step is one);
//  * each warp streams its digits through a ring in shared memory by asynchronous copies;
//  * global stores wait until the barrier has passed, and a reflector's root and reciprocals are
//    Newton steps;
//  * the kernel is kept small, since a column runs through all of it once: helpers are not
//    inlined, the product loop takes its plane half at run time and the loops that run once or
//    twice are not unrolled (108 KB -> 89 KB of code: stage `hetrd` of n = 305, 27 problems
//    5.8 -> 4.6 ms; peers' shared memory by 32-bit addresses, 77 KB: no faster; the product's units
//    taken by all 16 warps from a shared counter, 114 KB: 6.9 ms).
// A column is now bound by its chain of short phases (~7 us at n = 305), with one block per
// matrix by the stream of digits (16 B per entry and column: at n = 568, 128 problems, the
// first columns run at 4.6 to 4.8 TB/s of DRAM, 69 to 72 % of the measured rate).
// Measured (stage `hetrd` per step, ms, the FP64 panel's products -> now): n = 305, 27 problems
// 24.8 -> 4.6; n = 449, 40 problems 39.8 -> 10.6; n = 568, 2 problems 52 -> 9.9; 128 problems
// 79.3 -> 36.2; n = 2000, 1 problem 458 -> 89.
#include <cooperative_groups.h>
#include <cuda_fp16.h>

#include "nao_internal.cuh"
#include "reflector.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int HP_THREADS = 512;
constexpr int HP_MMA_WARPS = 8;                 // warps forming the digit products; the rest do FP64 work
constexpr int HP_FP_WARPS = HP_THREADS / 32 - HP_MMA_WARPS;
constexpr int HP_FP_THREADS = 32 * HP_FP_WARPS;
constexpr int HP_CHUNK = 32;                    // K steps (of 16 columns) of one exact FP32 sum
constexpr int HP_SLOTS = 16;                    // partial sums of the product's units
constexpr int HP_SLOTS2 = 24;                   // and of the panel's products
constexpr int HP_RED_WARPS = 4;
constexpr int NB = NAO_HT_NB;
constexpr int HD_S = 8;                         // digits per value of the FP64 form

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// q = round(x 2^{8S - 2 - e}) for |x| < 2^e (integer arithmetic on the bits of x)
template <int S>
__device__ __forceinline__ long long hd_fixed(double x, int e) {
  const long long bits = __double_as_longlong(x);
  const int b = (int)((bits >> 52) & 0x7ff);
  if (b == 0) return 0;
  long long m = (bits & 0xFFFFFFFFFFFFFll) | 0x10000000000000ll;
  const int sh = b - 1075 + 8 * S - 2 - e;
  long long q;
  if (sh >= 0) q = m << sh;
  else if (sh <= -62) q = 0;
  else q = (m + (1ll << (-sh - 1))) >> (-sh);
  return bits < 0 ? -q : q;
}

// S balanced base-256 digits d_s in [-128, 127] of q (|q| < 2^{8S-2}) as the bytes d_s + 128 of
// one word, least significant digit first: q + sum_k 128 256^k = sum_k (d_k + 128) 256^k
template <int S>
__device__ __forceinline__ unsigned long long hd_bytes(long long q) {
  return (unsigned long long)q + (0x8080808080808080ull >> (64 - 8 * S));
}
// byte of digit s (most significant first)
template <int S>
__device__ __forceinline__ unsigned int hd_byte(unsigned long long z, int s) {
  return (unsigned int)(z >> (8 * (S - 1 - s))) & 255u;
}
// four words' bytes b (0..3) gathered into one word
__device__ __forceinline__ unsigned int gather4(unsigned int a0, unsigned int a1, unsigned int a2, unsigned int a3, int b) {
  const unsigned int lo = __byte_perm(a0, a1, b | (b + 4) << 4), hi = __byte_perm(a2, a3, b | (b + 4) << 4);
  return __byte_perm(lo, hi, 0x5410);
}

// sum_{G < NG} R[G] 2^{-8 G} 2^ex as a double (NG <= 8), in integer arithmetic: the orders
// G < 4 and G >= 4 are combined exactly in two int64 words (|R[G]| < 2^31 gives |.| < 2^56
// each), which are then joined in one 63-bit integer, with a rounding of the low word far
// below the result's last bit, and converted with one rounding
template <int NG>
__device__ __forceinline__ double hd_combine(const int* R, int ex) {
  long long hi = 0, lo = 0;
#pragma unroll
  for (int G = 0; G < 4 && G < NG; ++G) hi += (long long)R[G] * (1ll << (8 * (3 - G)));
#pragma unroll
  for (int G = 4; G < NG; ++G) lo += (long long)R[G] * (1ll << (8 * (7 - G)));
  // value = (hi 2^32 + lo) 2^{ex - 56}; shift hi up by s <= 32 so that |hi 2^s| < 2^61
  const unsigned long long ah = hi < 0 ? 0ull - (unsigned long long)hi : (unsigned long long)hi;
  const int s = min(max(__clzll((long long)ah) - 3, 0), 32);
  long long t = (long long)((unsigned long long)hi << s);
  if (s == 32) t += lo;
  else t += (lo + (1ll << (31 - s))) >> (32 - s);
  return fix_to_double(t, ex - 56 - s + 32, false);
}

// (hi 2^32 + lo) 2^{ex - 56} for |hi| < 2^54, 0 <= lo < 2^54: the two words as orders.  Not inlined:
// a column runs through the whole kernel once, so the kernel has to fit in the instruction
// cache (with everything inlined it is 172 KB and every phase waits for instructions).
__device__ __noinline__ double hd_value(long long hi, long long lo, int ex) {
  const int R[HD_S] = {(int)(hi >> 24), 0, 0, (int)(hi & 0xFFFFFF), (int)(lo >> 24), 0, 0, (int)(lo & 0xFFFFFF)};
  return hd_combine<HD_S>(R, ex);
}

// element (r, c) of the Hermitian matrix stored as its lower triangle (column-major)
__device__ __forceinline__ z64 herm_at(const z64* A, int ld, int r, int c) {
  return c <= r ? A[(size_t)c * ld + r] : zconj(A[(size_t)r * ld + c]);
}

__host__ __device__ inline int hd_tiles(int n) { return n > 1 ? (n - 1 + 15) / 16 : 1; }

// Digit layout: tiles of 16 rows x 16 columns of the trailing matrix (rows and columns i0 + 1 ..),
// dig[p][row tile][column tile][q < S][lane] of 16 bytes, so that lane l = 4 g + t of a warp
// reads its part of the m16n8k16 A fragment: rows g and g + 8, columns 4 t .. 4 t + 3 (the
// fragment's k slots 2t, 2t + 1, 2t + 8, 2t + 9; B uses the same order).  Plane half h
// (planes h S/2 ..) lies in q = h S/2 .. h S/2 + S/2 - 1 as 2 S words: word
// row S + 2 (s - h S/2) + part holds the four columns' digits d + 128 as bytes.
// One block of eight warps per row tile: pass 1 takes each row's largest exponent, pass 2
// writes the digits.
template <int S>
__global__ void __launch_bounds__(256)
hetrd_digits_kernel(int n, const int32_t* __restrict__ size, const z64* __restrict__ Abase, int ld,
                    long long strideA, int i0, uint4* __restrict__ dig, int* __restrict__ erow) {
  const int p = blockIdx.y, T = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, g = lane >> 2, t = lane & 3;
  const int m = size ? size[p] : n;
  const int L = m - i0 - 1;
  if (16 * T >= L) return;  // uniform per block
  const z64* A = Abase + (size_t)p * strideA;
  const int NT = (L + 15) >> 4, NTn = hd_tiles(n);
  __shared__ int s_e[8][16];
  int bmax[2] = {0, 0};
  for (int k = wid; k < NT; k += 8) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int rr = 16 * T + g + 8 * h;
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        const int c = 16 * k + 4 * t + l;
        if (rr < L && c < L) {
          const z64 a = herm_at(A, ld, i0 + 1 + rr, i0 + 1 + c);
          bmax[h] = max(bmax[h], max(hd_exp(a.x), hd_exp(a.y)));
        }
      }
    }
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    bmax[h] = max(bmax[h], __shfl_xor_sync(0xffffffffu, bmax[h], 1));
    bmax[h] = max(bmax[h], __shfl_xor_sync(0xffffffffu, bmax[h], 2));
    if (t == 0) s_e[wid][g + 8 * h] = bmax[h];
  }
  __syncthreads();
  int e[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    int b = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) b = max(b, s_e[w][g + 8 * h]);
    e[h] = b == 0 ? -1100 : b - 1022;
    const int rr = 16 * T + g + 8 * h;
    if (wid == 0 && t == 0 && rr < L) erow[(size_t)p * (n > 1 ? n - 1 : 1) + rr] = e[h];
  }
  uint4* base = dig + ((size_t)p * NTn + T) * NTn * S * 32;
  for (int k = wid; k < NT; k += 8) {
    unsigned int w[2][2 * S];  // [plane half][row S + 2 sl + part]
#pragma unroll
    for (int row = 0; row < 2; ++row) {
      const int rr = 16 * T + g + 8 * row;
      unsigned long long z[2][4];
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        const int c = 16 * k + 4 * t + l;
        const z64 a = (rr < L && c < L) ? herm_at(A, ld, i0 + 1 + rr, i0 + 1 + c) : zmk(0.0, 0.0);
        z[0][l] = hd_bytes<S>(hd_fixed<S>(a.x, e[row]));
        z[1][l] = hd_bytes<S>(hd_fixed<S>(a.y, e[row]));
      }
#pragma unroll
      for (int part = 0; part < 2; ++part)
#pragma unroll
        for (int s = 0; s < S; ++s) {
          const int by = S - 1 - s;  // byte of digit s
          const int sh = by >= 4 ? 32 : 0;
          w[s / (S / 2)][row * S + 2 * (s % (S / 2)) + part] =
              gather4((unsigned int)(z[part][0] >> sh), (unsigned int)(z[part][1] >> sh),
                      (unsigned int)(z[part][2] >> sh), (unsigned int)(z[part][3] >> sh), by & 3);
        }
    }
    uint4* out = base + (size_t)k * S * 32 + lane;
#pragma unroll
    for (int q = 0; q < S; ++q) {
      const unsigned int* x = &w[q / (S / 2)][4 * (q % (S / 2))];
      out[q * 32] = make_uint4(x[0], x[1], x[2], x[3]);
    }
  }
}

// two digits (bytes u = d + 128 at positions sel of w) as packed f16 integers
__device__ __forceinline__ uint32_t hp_half2(uint32_t w, uint32_t sel) {
  const uint32_t x = __byte_perm(w, 0x64646464u, sel);  // 1024 + u each
  const __half2 h = __hsub2(*(const __half2*)&x, __half2{__ushort_as_half(0x6480), __ushort_as_half(0x6480)});  // - 1152
  return *(const uint32_t*)&h;
}

__device__ __forceinline__ void hp_mma(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// 16 bytes per lane and plane quarter from global to shared memory, asynchronously
template <int SH>
__device__ __forceinline__ void hp_copy(uint4* dst, const uint4* src) {
#pragma unroll
  for (int q = 0; q < SH; ++q)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                 :: "r"((uint32_t)__cvta_generic_to_shared(dst + q * 32)), "l"(src + q * 32) : "memory");
}

// Digit products of plane half H (0 or 1) of one 16-row tile over the K steps [k0, k1), added to
// (hi, lo)[4] (row g real, row g imaginary, row g + 8 real, imaginary) in units of 2^{-24} and
// 2^{-56}; per-lane partial sums (the caller adds the four lanes of a row).  K step k: the A
// digits at tile + k ts (S x 512 bytes), the B planes' 16 columns at bp + k bs (two parts of
// eight planes, PS halves apart).
// D > 0: every lane streams its own part of the A digits through a ring of D stages in shared
// memory (asynchronous copies, 2 KB per stage and warp, so that D K steps are in flight; a lane
// reads only what it copied itself, so no barrier is needed); D = 0: loads one step ahead.
template <int S, int D>
__device__ __forceinline__ void hp_tile_half(const uint4* tile, int ts, uint4* ring, const __half* bp, int bs, int PS,
                                             int k0, int k1, int H, int lane, long long* hi, long long* lo) {
  constexpr int SH = S / 2;  // planes of this half; also its uint4 per lane and K step
  const int g = lane >> 2, t = lane & 3;
  const __half* bre = bp + (size_t)g * PS + 4 * t;
  const __half* bim = bre + (size_t)8 * PS;
  const uint4* src = tile + H * SH * 32 + lane;
  uint4 nx[SH];
  if (D > 0) {
#pragma unroll
    for (int st = 0; st < D; ++st) {
      if (k0 + st < k1) hp_copy<SH>(ring + st * SH * 32 + lane, src + (size_t)(k0 + st) * ts);
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
  } else if (k0 < k1) {
#pragma unroll
    for (int q = 0; q < SH; ++q) nx[q] = src[(size_t)k0 * ts + q * 32];
  }
  int st = 0;
#pragma unroll 1
  for (int kc = k0; kc < k1; kc += HP_CHUNK) {
    const int ke = min(k1, kc + HP_CHUNK);
    float rr[SH][4], ri[SH][4];
#pragma unroll
    for (int s = 0; s < SH; ++s)
#pragma unroll
      for (int q = 0; q < 4; ++q) rr[s][q] = ri[s][q] = 0.0f;
#pragma unroll 1
    for (int k = kc; k < ke; ++k) {
      uint32_t w[4 * SH];
      if (D > 0) {
        asm volatile("cp.async.wait_group %0;" :: "n"(D > 0 ? D - 1 : 0) : "memory");
#pragma unroll
        for (int q = 0; q < SH; ++q) nx[q] = ring[(st * SH + q) * 32 + lane];
      }
#pragma unroll
      for (int q = 0; q < SH; ++q) {
        w[4 * q] = nx[q].x;
        w[4 * q + 1] = nx[q].y;
        w[4 * q + 2] = nx[q].z;
        w[4 * q + 3] = nx[q].w;
      }
      if (D > 0) {
        if (k + D < k1) hp_copy<SH>(ring + st * SH * 32 + lane, src + (size_t)(k + D) * ts);
        asm volatile("cp.async.commit_group;" ::: "memory");
        st = st + 1 == D ? 0 : st + 1;
      } else if (k + 1 < k1) {
#pragma unroll
        for (int q = 0; q < SH; ++q) nx[q] = src[(size_t)(k + 1) * ts + q * 32];
      }
      const uint2 br = *(const uint2*)(bre + (size_t)bs * k), bi = *(const uint2*)(bim + (size_t)bs * k);
      const uint32_t n0 = bi.x ^ 0x80008000u, n1 = bi.y ^ 0x80008000u;  // -Im
#pragma unroll
      for (int s = 0; s < SH; ++s) {
        uint32_t a[4];
        a[0] = hp_half2(w[2 * s], 0x4140);
        a[1] = hp_half2(w[S + 2 * s], 0x4140);
        a[2] = hp_half2(w[2 * s], 0x4342);
        a[3] = hp_half2(w[S + 2 * s], 0x4342);
        hp_mma(rr[s], a, br.x, br.y);
        hp_mma(ri[s], a, bi.x, bi.y);
        a[0] = hp_half2(w[2 * s + 1], 0x4140);
        a[1] = hp_half2(w[S + 2 * s + 1], 0x4140);
        a[2] = hp_half2(w[2 * s + 1], 0x4342);
        a[3] = hp_half2(w[S + 2 * s + 1], 0x4342);
        hp_mma(rr[s], a, n0, n1);
        hp_mma(ri[s], a, br.x, br.y);
      }
    }
    // R_st at lane 4 g + t', columns 2 t' + e: order s + e + b with b = SH H + 2 t'; the eight
    // sums of a row and part meet in one 57-bit integer q (units of 2^{-32 - 8 b})
    const int sft = 8 + 8 * (SH * H + 2 * t);
    if (sft < 64) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        long long q = 0;
#pragma unroll
        for (int s = 0; s < SH; ++s) {
          const float* f = (c & 1) ? ri[s] : rr[s];
          q += (long long)__float2int_rn(f[c & 2]) * (1ll << (8 * (4 - s)));
          q += (long long)__float2int_rn(f[(c & 2) + 1]) * (1ll << (8 * (3 - s)));
        }
        hi[c] += q >> sft;
        const unsigned long long rem = (unsigned long long)q << (64 - sft);  // the bits below, at the top
        lo[c] += (long long)(rem >> 32);
      }
    }
  }
}

__device__ __forceinline__ long long add_quad(long long v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// The plane halves [h0, h1) of one tile; lane 4 g + tq returns (hi, lo) of its combination tq:
// row g + 8 (tq >> 1), part tq & 1.
// Not inlined: the product loop then has the registers to itself, and the kernel's pointers are
// saved once per unit.
template <int S, int D>
__device__ __noinline__ longlong2 hp_unit(const uint4* tile, int ts, uint4* ring, const __half* bp, int bs, int PS,
                                             int k0, int k1, int h0, int h1, int lane) {
  long long hi[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};
#pragma unroll 1
  for (int h = h0; h < h1; ++h) hp_tile_half<S, D>(tile, ts, ring, bp, bs, PS, k0, k1, h, lane, hi, lo);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    hi[c] = add_quad(hi[c]);
    lo[c] = add_quad(lo[c]);
  }
  const int tq = lane & 3;
  return make_longlong2(tq == 0 ? hi[0] : tq == 1 ? hi[1] : tq == 2 ? hi[2] : hi[3],
                        tq == 0 ? lo[0] : tq == 1 ? lo[1] : tq == 2 ? lo[2] : lo[3]);
}

// Global copies of panel column jj (own rows): V below the subdiagonal of A's column (Procedure 3)
// and the rows of VWr.  They are written while the next column is under way: a cluster barrier
// with stores to global memory outstanding takes ~4000 cycles instead of ~500.
__device__ __noinline__ void store_column(z64* __restrict__ Acol, z64* __restrict__ VWrow, const z64* v, const z64* wown,
                                          int jj, double beta, int C, int rank, int Rown, int Lp, int t0, int nt) {
#pragma unroll 1
  for (int lr = t0; lr < Rown; lr += nt) {
    const int r = ((lr >> 4) * C + rank) * 16 + (lr & 15);
    if (r < jj || r >= Lp) continue;
    const z64 vr = v[lr], wr = wown[lr];
    Acol[r] = r == jj ? zmk(beta, 0.0) : vr;
    z64* o = VWrow + (size_t)r * 3 * NB + jj;
    o[0] = vr;
    o[2 * NB] = vr;
    o[NB] = wr;
  }
}

// sum of `per` slots, 32 apart
__device__ __forceinline__ longlong2 hp_sum(const longlong2* s, int per) {
  longlong2 h = make_longlong2(0, 0);
#pragma unroll 1
  for (int q = 0; q < per; ++q) {
    h.x += s[q * 32].x;
    h.y += s[q * 32].y;
  }
  return h;
}

// Word of an eight-plane digit tile (one K step, 4 KB) that holds plane s and part of row `row`
// (0..15) for the columns 4 t .. 4 t + 3: at hp_base + hp_plane(s)
__device__ __forceinline__ unsigned char* hp_base(uint4* tile, int row, int t, int part) {
  return (unsigned char*)tile + (row >> 3) * 1024 + (row & 7) * 64 + t * 16 + part * 4;
}
__device__ __forceinline__ constexpr int hp_plane(int s) { return (s >> 2) * 2048 + ((s & 3) >> 1) * 512 + (s & 1) * 8; }

// digits of val 2^{-ex} as f16, the planes st halves apart
__device__ __noinline__ void hp_put(__half* o, int st, double val, int ex) {
  const unsigned long long z = hd_bytes<8>(hd_fixed<8>(val, ex));
  const unsigned int hi = (unsigned int)(z >> 32), lo = (unsigned int)z;
#pragma unroll
  for (int s = 0; s < 8; s += 2) {  // planes s (the higher byte) and s + 1
    const uint32_t h = hp_half2(s < 4 ? hi : lo, (s & 2) ? 0x4041 : 0x4243);
    o[(size_t)s * st] = __ushort_as_half((unsigned short)h);
    o[(size_t)(s + 1) * st] = __ushort_as_half((unsigned short)(h >> 16));
  }
}

// Shared-memory layout (units of 16 bytes from the start), common to host and device.
constexpr int HP_TILE = 256;         // uint4 of one eight-plane digit tile
constexpr int HP_MDT = 4 * HP_TILE;  // of an own row tile's panel digits (64 columns), one orientation
constexpr int HP_PS = 64 + 16;       // halves between two digit planes of the 64 coefficients
struct PanelSmem {
  int x, v, p, un, w, cf, cr, yp, ys, slots, vd, cd, ring, md;
  int PS;           // halves between two digit planes of v (16 mod 64: conflict-free fragment reads)
  int own;          // own row tiles of a block
  bool md_in_smem;  // the panel's digit tiles
  size_t bytes;
};

// shared: x lies in the first half of vd (the real part's digits).  The digits are dead once every
// block has formed its products (B2), which is before the next column is pushed, and v's digits
// are formed from x through a copy of its real parts in the rings, which are idle then.
__host__ __device__ inline PanelSmem panel_smem(int n, int C, int D, size_t limit, bool shared) {
  PanelSmem s;
  const int NT = hd_tiles(n);
  s.own = (NT + C - 1) / C;
  const int R = 16 * s.own;
  s.PS = (16 * NT + 63) / 64 * 64 + 16;
  int o = 0;
  s.x = o, o += shared ? 0 : 16 * NT;
  s.v = o, o += R;
  s.p = o, o += R;
  s.un = o, o += R;
  s.w = o, o += R;
  s.cf = o, o += 2 * 2 * NB;
  s.cr = o, o += 2 * NB;
  s.yp = o, o += 2 * NB;
  s.ys = o, o += 2 * NB;
  s.slots = o, o += (HP_SLOTS + HP_SLOTS2) * 32;
  s.vd = o, o += 2 * s.PS;
  if (shared) s.x = s.vd;
  s.cd = o, o += 2 * 2 * HP_PS;
  s.ring = o, o += HP_MMA_WARPS * D * 128;  // (of every warp when the panel's digits come from global memory)
  s.md = o;
  s.md_in_smem = (size_t)(o + 2 * s.own * HP_MDT) * 16 <= limit;
  o += s.md_in_smem ? 2 * s.own * HP_MDT : HP_FP_WARPS * D * 128;
  s.bytes = (size_t)o * 16;
  return s;
}

constexpr size_t HP_SMEM_LIMIT = 225 * 1024;  // of 227 KB: the kernel's static arrays take the rest

// One panel.  MDbase: scratch for the blocks' panel digits where they do not fit in shared
// memory; VWr: the panel's [V | W | V] rows (row-major, 3 NB columns) for the update product.
//
// Panel digits: column c = 2 jj + (0: V, 1: W) of the panel, split like v with a power-of-two
// scale (V: 2; W: 2^{s_wx[jj]}, of the block's own rows), as two sets of tiles per own row tile lt:
//   md1[lt][c >> 4]  rows c & 15, columns the tile's 16 trailing rows, holding conj(M): the
//                    A operand of y = M^H v (the contraction runs over the own row tiles);
//   md2[lt][c >> 4]  rows the tile's trailing rows, columns c & 15: the A operand of
//                    M coef (the contraction runs over the panel's columns).
// Bytes not written yet are digits of finite values that meet zero coefficients or rows that
// nothing reads.
template <int S, int D, bool SHARED>
__global__ void __launch_bounds__(HP_THREADS, 1)
hetrd_panel_mma_kernel(int n, const int32_t* __restrict__ size, z64* __restrict__ Abase, int ld, long long strideA,
                       double* __restrict__ dbase, double* __restrict__ ebase, z64* __restrict__ taubase,
                       long long strideV, int i0, const uint4* __restrict__ dig, const int* __restrict__ erowbase,
                       uint4* __restrict__ MDbase, z64* __restrict__ VWrbase, long long strideVW) {
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int rc = (65536 + C - 1) / C;  // t / C = t rc >> 16 for the tile counts t <= 256
  extern __shared__ z64 sm[];
  __shared__ z64 s_tau, s_scale, s_w0, s_c0, s_p0;
  __shared__ double s_beta, s_diag, s_alpha2, s_yy, s_delta;
  __shared__ double red[8], aw[HP_MMA_WARPS];
  __shared__ int s_wx[NB];  // exponent of W's column jj over the own rows (|w| < 2^s_wx)
  __shared__ int s_cx[2];   // exponents (+ 8192; 0: none) of the scaled coefficients: next column, corrections
  const int p = blockIdx.x / C;
  const int m = size ? size[p] : n;
  const int Lp = m - i0 - 1;  // trailing rows at the panel's start
  if (Lp < 0) return;         // uniform over the cluster
  z64* A = Abase + (size_t)p * strideA;
  double* d = dbase + (size_t)p * strideV;
  double* e = ebase + (size_t)p * strideV;
  z64* tau = taubase + (size_t)p * strideV;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (Lp == 0) {  // only the last diagonal element
    if (rank == 0 && tid == 0) {
      d[m - 1] = A[(size_t)(m - 1) * ld + (m - 1)].x;
      e[m - 1] = 0.0;
      tau[m - 1] = zmk(0.0, 0.0);
    }
    return;
  }
  const PanelSmem L = panel_smem(n, C, D, HP_SMEM_LIMIT, SHARED);
  z64 *x = sm + L.x, *v = sm + L.v, *pown = sm + L.p, *unext = sm + L.un, *wown = sm + L.w, *coefs = sm + L.cf,
      *crow = sm + L.cr, *ypart = sm + L.yp, *ysum = sm + L.ys;
  longlong2* slots = (longlong2*)(sm + L.slots);  // of the MMA warps, then of the others
  __half* vd = (__half*)(sm + L.vd);
  __half* cd = (__half*)(sm + L.cd);  // digits of the coefficients: next column, corrections
  const int PS = L.PS;
  uint4* ring = (uint4*)(sm + L.ring) + wid * D * 128;
  z64* VWr = VWrbase + (size_t)p * strideVW;
  auto div_c = [&](int t) { return t * rc >> 16; };
  const int NT = (Lp + 15) >> 4, NTn = hd_tiles(n);
  const int nown = NT > rank ? div_c(NT - rank + C - 1) : 0;  // own row tiles rank, rank + C, ...
  const int Rown = 16 * nown;
  uint4* md1 = L.md_in_smem ? (uint4*)(sm + L.md) : MDbase + ((size_t)p * C + rank) * 2 * L.own * HP_MDT;
  uint4* md2 = md1 + (size_t)L.own * HP_MDT;
  const uint4* digp = dig + (size_t)p * NTn * NTn * S * 32;
  const int* erow = erowbase + (size_t)p * (n > 1 ? n - 1 : 1);
  const int iend = min(i0 + NB, m);
  auto csync = [&]() {
    if (C == 1) __syncthreads();
    else cluster.sync();
  };
  // trailing row of local row lr; exponent of panel column c's scale
  auto row_of = [&](int lr) { return ((lr >> 4) * C + rank) * 16 + (lr & 15); };
  auto col_exp = [&](int c) { return (c & 1) ? s_wx[c >> 1] : 1; };
  // a unit of the panel's products (D stages ahead from global memory)
  auto panel_unit = [&](const uint4* tile, int ts, const __half* bp, int bs, int ps, int k0, int k1, int h0, int h1) {
    return L.md_in_smem ? hp_unit<8, 0>(tile, ts, nullptr, bp, bs, ps, k0, k1, h0, h1, lane)
                        : hp_unit<8, D>(tile, ts, ring, bp, bs, ps, k0, k1, h0, h1, lane);
  };
  // this lane's (row, part) of a unit's result
  const int urow = (lane >> 2) + 8 * ((lane >> 1) & 1), upart = lane & 1;

#pragma unroll 1
  for (int r = tid; r < Lp; r += HP_THREADS) x[r] = A[(size_t)i0 * ld + i0 + 1 + r];
#pragma unroll 1
  for (int r = tid; r < 2 * 2 * HP_PS; r += HP_THREADS) sm[L.cd + r] = zmk(0.0, 0.0);
  if (tid == 0) s_diag = A[(size_t)i0 * ld + i0].x;
  if (tid < NB) s_wx[tid] = -1100;
  if (tid < 2) s_cx[tid] = 0;
  csync();  // (the other blocks' shared memory exists from here on)

  double beta_prev = 0.0;
  int jlast = -1;  // last column whose global copies are still to be written
#pragma unroll 1
  for (int i = i0; i < iend; ++i) {
    const int j = i - i0;  // trailing rows j .. Lp - 1 hold x = A(i + 1 :, i)
    if (j == Lp) {  // last diagonal element, no reflector
      if (rank == 0 && tid == 0) {
        d[i] = s_diag;
        e[i] = 0.0;
        tau[i] = zmk(0.0, 0.0);
      }
      break;
    }
    const z64* cf = coefs + (j & 1) * 2 * NB;  // conj(M(i + 1, c ^ 1)), c < 2 j
    z64* cfn = coefs + ((j + 1) & 1) * 2 * NB;
    const int nq = (j + 7) >> 3;  // tiles of the panel columns c < 2 j
    const int ks0 = j >> 4;
    const int lt0 = ks0 > rank ? div_c(ks0 - rank + C - 1) : 0;  // first own tile with live rows
    const int lr0 = 16 * lt0, nl = max(nown - lt0, 0);
    // ---- Procedures 1-2, in every block: the norm of x(1:) in four warps; the others write the
    // digits of panel column j - 1
    if (wid < HP_RED_WARPS) {
      double s = 0.0;
#pragma unroll 1
      for (int r = j + 1 + tid; r < Lp; r += 32 * HP_RED_WARPS) s += zabs2(x[r]);
      s = warp_sum(s);
      if (lane == 0) red[wid] = s;
    } else if (j > 0) {
      const int jj = j - 1;
#pragma unroll 1
      for (int it = tid - 32 * HP_RED_WARPS; it < 4 * Rown; it += HP_THREADS - 32 * HP_RED_WARPS) {
        const int part = it & 1, vw = (it >> 1) & 1, lr = it >> 2, r = row_of(lr), c = 2 * jj + vw, row = lr & 15;
        const double val = (r >= jj && r < Lp) ? ((const double*)((vw ? wown : v) + lr))[part] : 0.0;
        const long long fx = hd_fixed<8>(val, vw ? s_wx[jj] : 1);
        const unsigned long long z = hd_bytes<8>(fx), zc = part ? hd_bytes<8>(-fx) : z;  // md1 holds conj(M)
        const int to = (lr >> 4) * HP_MDT + (c >> 4) * HP_TILE;
        unsigned char* b1 = hp_base(md1 + to, c & 15, row >> 2, part) + (row & 3);
        unsigned char* b2 = hp_base(md2 + to, row, (c & 15) >> 2, part) + (c & 3);
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          b1[hp_plane(s)] = (unsigned char)hd_byte<8>(zc, s);
          b2[hp_plane(s)] = (unsigned char)hd_byte<8>(z, s);
        }
      }
    }
    __syncthreads();
    if (tid == 0) {
      z64 t, scale;
      double beta;
      reflector(x[j], (red[0] + red[1]) + (red[2] + red[3]), t, scale, beta);
      s_tau = t;
      s_scale = scale;
      s_beta = beta;
    } else if (wid == 1) {
      // exponent of the next column's coefficients, scaled by the columns' exponents
      int bm = 0;
#pragma unroll 1
      for (int c = lane; c < 2 * j; c += 32) {
        const z64 a = cf[c];
        const int b = max(hd_exp(a.x), hd_exp(a.y));
        if (b) bm = max(bm, b - 1022 + col_exp(c) + 8192);
      }
      bm = __reduce_max_sync(0xffffffffu, bm);
      if (lane == 0) {
        s_cx[0] = bm;
        s_cx[1] = 0;
      }
    } else if (j > 0 && wid >= HP_RED_WARPS) {
      store_column(A + (size_t)(i - 1) * ld + i0 + 1, VWr + (size_t)(i0 + 1) * 3 * NB, v, wown, j - 1, beta_prev, C, rank, Rown,
                   Lp, tid - 32 * HP_RED_WARPS, HP_THREADS - 32 * HP_RED_WARPS);
    }
    __syncthreads();
    const z64 t = s_tau, scale = s_scale;
    const bool active = !(t.x == 0.0 && t.y == 0.0);  // H_i = I otherwise (uniform)
    beta_prev = s_beta;
    jlast = j;
    if (rank == 0 && tid == HP_THREADS - 1) {
      d[i] = s_diag;
      e[i] = s_beta;
      tau[i] = t;
    }
    // v = x / (alpha - beta), its digit planes (|v| <= 1 < 2), and v of the own rows
#pragma unroll 1
    for (int it = tid; it < 32 * (NT - ks0); it += HP_THREADS) {
      const int r = 16 * ks0 + (it >> 1), part = it & 1;
      double val = 0.0;
      if (r == j) {
        val = part ? 0.0 : 1.0;
      } else if (r > j && r < Lp) {
        const z64 xr = x[r];
        val = part ? fma(xr.x, scale.y, xr.y * scale.x) : fma(xr.x, scale.x, -(xr.y * scale.y));
      }
      const int lt = div_c(r >> 4);
      if (lt * C + rank == r >> 4) ((double*)&v[16 * lt + (r & 15)])[part] = active ? val : 0.0;
      if (SHARED && part == 0) ((double*)(sm + L.ring))[r] = val;  // (x is still being read)
      else hp_put(vd + (size_t)part * 8 * PS + r, PS, val, 1);
    }
    if (SHARED) {
      __syncthreads();
#pragma unroll 1
      for (int r = 16 * ks0 + tid; r < 16 * NT; r += HP_THREADS) hp_put(vd + r, PS, ((const double*)(sm + L.ring))[r], 1);
    }
    if (tid >= HP_THREADS - 128) {  // the next column's coefficients' digits
      const int c = (tid & 127) >> 1, part = tid & 1;
      if (c < 2 * j) hp_put(cd + (size_t)part * 8 * HP_PS + c, HP_PS, part ? cf[c].y : cf[c].x, s_cx[0] - 8192 - col_exp(c));
    }
    __syncthreads();
    const bool more = j + 1 < NB && i + 1 < iend;  // the panel has a next column
    longlong2* sl = slots + HP_SLOTS * 32;
    auto fsync = [] { asm volatile("bar.sync 1, %0;" :: "n"(HP_FP_THREADS) : "memory"); };

    // ---- Procedure 4: p = A22 v of the own rows, from the digits; a tile per unit, or with
    // few tiles (tile, K segment, plane half)
    const int nk = NT - ks0;
    const bool tiles = nl >= HP_MMA_WARPS;
    int lsegs = 0;
    if (!tiles) {
      int best = 1 << 30;
#pragma unroll 1
      for (int q = 0; (2 * nl << q) <= HP_SLOTS && (1 << q) <= nk; ++q) {
        const int cost = ((2 * nl << q) + HP_MMA_WARPS - 1) / HP_MMA_WARPS * ((nk >> q) + 5);
        if (cost < best) best = cost, lsegs = q;
      }
    }
    const int lper = tiles ? 0 : lsegs + 1;  // log2 of the units per tile
    double dacc = 0.0;  // this lane's part of Re(p^H v)
    auto finish = [&](int lt, longlong2 h) {
      const int r = 16 * (lt * C + rank) + urow;
      if (r < j || r >= Lp) return;
      const double pv = hd_value(h.x, h.y, erow[r] + 1 - 12);
      ((double*)&pown[16 * lt + urow])[upart] = pv;
      dacc = fma(pv, ((const double*)&v[16 * lt + urow])[upart], dacc);
    };
    if (wid >= HP_MMA_WARPS) {
      // ---- the panel's products
      const int fw = wid - HP_MMA_WARPS;
      if (more && fw == HP_FP_WARPS - 1 && j + 1 < Lp && rank == ((j + 1) >> 4) - C * div_c((j + 1) >> 4)) {
        // the panel's row i + 2 so far: the coefficients of the column after the next
#pragma unroll 1
        for (int c = lane; c < 2 * j; c += 32)
          crow[c] = __ldcg(VWr + (size_t)(i0 + 2 + j) * 3 * NB + (c & 1) * NB + (c >> 1));
      }
      // y = M^H v over the own rows, (tile of columns, plane half) per unit, and column i + 1's
      // updates by panel columns 0 .. j-1, a tile or (tile, plane half) per unit
      const bool whole = nl >= HP_FP_WARPS;
      const int ny = active && j > 0 ? nq : 0, nx = more ? nl : 0;
      auto next_at = [&](int lt) -> double {  // this lane's part of column i + 1 so far
        const int r = 16 * (lt * C + rank) + urow;
        return r >= j && r < Lp ? ((const double*)&A[(size_t)(i + 1) * ld + i0 + 1 + r])[upart] : 0.0;
      };
      auto next_put = [&](int lt, double a, longlong2 h) {
        ((double*)&unext[16 * lt + urow])[upart] = j > 0 ? a - hd_value(h.x, h.y, s_cx[0] - 8192 - 12) : a;
      };
      if (j == 0) {
#pragma unroll 1
        for (int q = fw; q < nx; q += HP_FP_WARPS) next_put(lt0 + q, next_at(lt0 + q), make_longlong2(0, 0));
      } else {
        double a0[2] = {0.0, 0.0};  // (slot mode: a warp finishes at most two tiles)
        if (!whole)
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int u = fw + q * HP_FP_WARPS - ny;
            if (u >= 0 && u < nx) a0[q] = next_at(lt0 + u);
          }
#pragma unroll 1
        for (int u = fw; u < 2 * ny + (whole ? nx : 2 * nx); u += HP_FP_WARPS) {
          const bool isy = u < 2 * ny;
          const int w = isy ? u : u - 2 * ny;
          const int lt = lt0 + (whole ? w : w >> 1);
          const double a = !isy && whole ? next_at(lt) : 0.0;
          const longlong2 h = panel_unit(isy ? md1 + (w >> 1) * HP_TILE : md2 + (size_t)lt * HP_MDT,
                                         isy ? HP_MDT : HP_TILE, isy ? vd + 16 * rank : cd, isy ? 16 * C : 16,
                                         isy ? PS : HP_PS, isy ? lt0 : 0, isy ? nown : nq,
                                         isy || !whole ? w & 1 : 0, isy || !whole ? (w & 1) + 1 : 2);
          if (!isy && whole) next_put(lt, a, h);
          else sl[u * 32 + lane] = h;
        }
        fsync();
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int q = fw + k * HP_FP_WARPS;
          if (q < ny) {
            const longlong2 h = hp_sum(sl + 2 * q * 32 + lane, 2);
            const int c = 16 * q + urow;
            if (c < 2 * j) ((double*)&ypart[c])[upart] = hd_value(h.x, h.y, col_exp(c) + 1 - 12);
          } else if (!whole && q - ny < nx) {
            next_put(lt0 + q - ny, a0[k], hp_sum(sl + 2 * q * 32 + lane, 2));
          }
        }
      }
    }
    if (wid < HP_MMA_WARPS) {
      if (active) {
#pragma unroll 1
        for (int u = wid; u < nl << lper; u += HP_MMA_WARPS) {
          const int lt = lt0 + (u >> lper), w = u - ((u >> lper) << lper), sg = w >> 1;
          const longlong2 h =
              hp_unit<S, D>(digp + (size_t)(lt * C + rank) * NTn * S * 32, S * 32, ring, vd, 16, PS, ks0 + (sg * nk >> lsegs),
                            ks0 + ((sg + 1) * nk >> lsegs), tiles ? 0 : w & 1, tiles ? 2 : (w & 1) + 1, lane);
          if (tiles) finish(lt, h);
          else slots[u * 32 + lane] = h;
        }
        if (!tiles) {
          asm volatile("bar.sync 2, %0;" :: "n"(32 * HP_MMA_WARPS) : "memory");
#pragma unroll 1
          for (int q = wid; q < nl; q += HP_MMA_WARPS) finish(lt0 + q, hp_sum(slots + (q << lper) * 32 + lane, 1 << lper));
        }
      }
      dacc = warp_sum(dacc);
      if (lane == 0) aw[wid] = dacc;
    }
    if (C > 1) cluster.sync();  // B2: partial sums ready
    // y = M^H v of all blocks summed (fixed order) and what follows from it: Re(y1^H y2), the
    // correction of trailing row j, and the own rows' corrections sum_c M(r, c) y(c ^ 1), into
    // the slots (fewer tiles than warps) or wown; by all warps, or with one block by the panel
    // warps beside the digit products
    const int nwc = C == 1 ? HP_FP_WARPS : HP_THREADS / 32, cw = wid - (C == 1 ? HP_MMA_WARPS : 0);
    longlong2* slc = C == 1 ? sl : slots;
    if (active && cw >= 0) {
      auto wsync = [&] { asm volatile("bar.sync %0, %1;" :: "r"(C == 1 ? 1 : 4), "r"(32 * nwc) : "memory"); };
      const int ct = 32 * cw + lane;
      if (j > 0) {
        if (C == 1) wsync();
        if (ct < 4 * j) {  // (column, part) per thread
          const int c = ct >> 1, part = ct & 1;
          double a = 0.0;
          for (int k = 0; k < C; k += 8) {  // eight remote loads in flight
            double b[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
              b[q] = k + q < C ? ((const double*)&cluster.map_shared_rank(ypart, k + q)[c])[part] : 0.0;
            a += ((b[0] + b[1]) + (b[2] + b[3])) + ((b[4] + b[5]) + (b[6] + b[7]));
          }
          ((double*)&ysum[c])[part] = a;
          const int b = hd_exp(a);
          if (b) atomicMax(&s_cx[1], b - 1022 + col_exp(c ^ 1) + 8192);
        }
        wsync();
        if (ct < 4 * j) {
          const int c = ct >> 1, part = ct & 1;
          hp_put(cd + (size_t)(16 + part * 8) * HP_PS + (c ^ 1), HP_PS, ((const double*)&ysum[c])[part],
                 s_cx[1] - 8192 - col_exp(c ^ 1));
        } else if (cw == 7) {
          double a = 0.0;
          if (lane < j) {
            const z64 y2 = ysum[2 * lane], y1 = ysum[2 * lane + 1];
            a = fma(y1.x, y2.x, y1.y * y2.y);
          }
          a = warp_sum(a);
          if (lane == 0) s_yy = a;
        } else if (cw == 5 || cw == 6) {  // V(i+1, :) y1 + W(i+1, :) y2 = sum_c conj(cf) y
          double a = 0.0;
          for (int c = lane; c < 2 * j; c += 32) {
            const z64 f = cf[c], y = ysum[c];
            a = cw == 5 ? fma(f.x, y.y, fma(-f.y, y.x, a)) : fma(f.x, y.x, fma(f.y, y.y, a));
          }
          a = warp_sum(a);
          if (lane == 0) ((double*)&s_c0)[cw == 5] = a;
        }
      }
      if (C > 1) {  // the blocks' sums of Re(p_raw^H v), and p_raw of trailing row j
        if (cw == 8) {
          double a = 0.0;
#pragma unroll
          for (int q = 0; q < 16 * HP_MMA_WARPS / 32; ++q) {
            const int k = lane + 32 * q;
            if (k < C * HP_MMA_WARPS) a += cluster.map_shared_rank(aw, k / HP_MMA_WARPS)[k % HP_MMA_WARPS];
          }
          a = warp_sum(a);
          if (lane == 0) s_delta = a;
        } else if (cw == 9 && lane == 0) {
          const int q = div_c(ks0);
          s_p0 = cluster.map_shared_rank(pown, ks0 - C * q)[16 * q + (j & 15)];
        }
      }
      if (j > 0 || C > 1) wsync();
      if (j > 0) {
        const bool whole = nl >= nwc;
        for (int u = cw; u < (whole ? nl : 2 * nl); u += nwc) {
          const int lt = lt0 + (whole ? u : u >> 1);
          const longlong2 h = panel_unit(md2 + (size_t)lt * HP_MDT, HP_TILE, cd + 16 * HP_PS, 16, HP_PS, 0, nq,
                                         whole ? 0 : u & 1, whole ? 2 : (u & 1) + 1);
          if (whole) ((double*)&wown[16 * lt + urow])[upart] = hd_value(h.x, h.y, s_cx[1] - 8192 - 12);
          else slc[u * 32 + lane] = h;
        }
      }
    }
    if (C == 1) __syncthreads();  // B2
    // ---- Procedure 5: w = tau p - (|tau|^2 / 2) (p^H v) v with the corrected p.  The last warp
    // forms p^H v = p_raw^H v - 2 Re(y1^H y2) and w of trailing row j (where v = 1)
    if (active && tid == HP_THREADS - 32) {
      double a;
      z64 p0;
      if (C > 1) {
        a = s_delta;
        p0 = s_p0;
      } else {
        a = ((aw[0] + aw[1]) + (aw[2] + aw[3])) + ((aw[4] + aw[5]) + (aw[6] + aw[7]));
        p0 = pown[j];
      }
      if (j > 0) {
        a = fma(-2.0, s_yy, a);
        p0 = zsub(p0, s_c0);
      }
      const double a2 = -0.5 * zabs2(t) * a;
      const z64 q = zmul(t, p0);
      s_alpha2 = a2;
      s_w0 = zmk(q.x + a2, q.y);
    }
    __syncthreads();
    // ---- W of the own rows, and their share of the next column, pushed to every block
    {
      const z64 w0 = active ? s_w0 : zmk(0.0, 0.0);
      const double a2 = active ? s_alpha2 : 0.0;
      const bool whole = nl >= nwc;
      int wx = 0;
#pragma unroll 1
      for (int b = 2 * lr0; b < 2 * Rown; b += HP_THREADS) {  // (row, part) per thread
        const int lr = (b + tid) >> 1, part = tid & 1, r = row_of(lr);
        const bool live = lr < Rown && r >= j && r < Lp;
        double pr = 0.0, vp = 0.0, vo = 0.0, un = 0.0;
        if (live) {
          vp = ((const double*)&v[lr])[part];
          vo = ((const double*)&v[lr])[part ^ 1];
          if (more) un = ((const double*)&unext[lr])[part];
          if (active) {
            pr = ((const double*)&pown[lr])[part];
            if (j > 0) {
              if (whole) {
                pr -= ((const double*)&wown[lr])[part];
              } else {  // lane 4 (row & 7) + 2 (row >> 3) + part of the tile's two slots
                const longlong2 h = hp_sum(slc + ((lr >> 4) - lt0) * 64 + 4 * (lr & 7) + 2 * ((lr >> 3) & 1) + part, 2);
                pr -= hd_value(h.x, h.y, s_cx[1] - 8192 - 12);
              }
            }
          }
        }
        const double po = __shfl_xor_sync(0xffffffffu, pr, 1);
        const double wr = fma(t.x, pr, fma(part ? t.y : -t.y, po, a2 * vp));
        if (!live) continue;
        ((double*)&wown[lr])[part] = wr;
        wx = max(wx, hd_exp(wr));
        if (more) {  // - V(r, j) conj(W(i + 1, j)) - W(r, j) conj(V(i + 1, j)), V(i + 1, j) = 1 (0 when H_i = I)
          const double xn = fma(-vp, w0.x, fma(part ? vo : -vo, w0.y, un)) - wr;
#pragma unroll 1
          for (int k = 0; k < C; ++k) {
            if (r != j) ((double*)&cluster.map_shared_rank(x, k)[r])[part] = xn;
            else if (part == 0) *cluster.map_shared_rank(&s_diag, k) = xn;
          }
          if (r == j + 1)
#pragma unroll 1
            for (int k = 0; k < C; ++k) {
              double* cn = (double*)(cluster.map_shared_rank(cfn, k) + 2 * j) + part;
              cn[0] = part ? -wr : wr;
              cn[2] = part ? -vp : vp;
            }
        }
      }
      wx = __reduce_max_sync(0xffffffffu, wx);
      if (lane == 0 && wx) atomicMax(&s_wx[j], wx - 1022);
    }
    if (more && j + 1 < Lp && rank == ((j + 1) >> 4) - C * div_c((j + 1) >> 4) && wid == HP_THREADS / 32 - 1)
#pragma unroll 1
      for (int c = lane; c < 2 * j; c += 32)
#pragma unroll 1
        for (int k = 0; k < C; ++k) cluster.map_shared_rank(cfn, k)[c ^ 1] = zconj(crow[c]);
    csync();  // B1: column i + 1 is in every block's shared memory
  }
  if (jlast >= 0)  // the last column's global copies
    store_column(A + (size_t)(i0 + jlast) * ld + i0 + 1, VWr + (size_t)(i0 + 1) * 3 * NB, v, wown, jlast, beta_prev, C, rank,
                 Rown, Lp, tid, HP_THREADS);
}

int smem_optin() {
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return optin;
}

constexpr int HP_MAX_CLUSTER = 16;  // (beyond 8: the non-portable size)

// Form of a panel at order n with C blocks a matrix: stages of the rings (four, or two where that makes
// room for the panel's digits or for the vectors of a large matrix; 0: does not fit), and whether x
// lies in vd's space, where there is no room for both.
struct PanelForm {
  int D;
  bool shared;
};

PanelForm panel_form(int n, int C) {
  const PanelSmem s4 = panel_smem(n, C, 4, HP_SMEM_LIMIT, false), s2 = panel_smem(n, C, 2, HP_SMEM_LIMIT, false);
  if (s4.md_in_smem) return {4, false};
  if (s2.md_in_smem) return {2, false};
  if (s4.bytes <= HP_SMEM_LIMIT) return {4, false};
  if (s2.bytes <= HP_SMEM_LIMIT) return {2, false};
  return {panel_smem(n, C, 2, HP_SMEM_LIMIT, true).bytes <= HP_SMEM_LIMIT ? 2 : 0, true};
}

typedef void (*PanelFn)(int, const int32_t*, z64*, int, long long, double*, double*, z64*, long long, int, const uint4*,
                        const int*, uint4*, z64*, long long);

template <int S>
PanelFn panel_fn_s(PanelForm f) {
  if (f.shared) return hetrd_panel_mma_kernel<S, 2, true>;
  return f.D == 4 ? hetrd_panel_mma_kernel<S, 4, false> : hetrd_panel_mma_kernel<S, 2, false>;
}

PanelFn panel_fn(int digits, PanelForm f) { return digits == 6 ? panel_fn_s<6>(f) : panel_fn_s<HD_S>(f); }

cudaError_t panel_config(PanelFn fn, cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int n, int nprob, int C, PanelForm f,
                         cudaStream_t st) {
  cfg.gridDim = dim3((unsigned)(nprob * C));
  cfg.blockDim = dim3(HP_THREADS);
  cfg.dynamicSmemBytes = panel_smem(n, C, f.D, HP_SMEM_LIMIT, f.shared).bytes;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)HP_SMEM_LIMIT);
  if (err == cudaSuccess) err = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return err;
}

}  // namespace

bool hetrd_digits_fit(int n, int digits) {
  (void)digits;
  return panel_form(n, HP_MAX_CLUSTER).D > 0 && (size_t)smem_optin() >= HP_SMEM_LIMIT + 1024;
}

size_t hetrd_panel_bytes(int n, int nprob) {
  const int NT = hd_tiles(n);
  if (panel_smem(n, 1, 2, HP_SMEM_LIMIT, false).md_in_smem) return 16;  // (also with more blocks)
  return (size_t)(NT + HP_MAX_CLUSTER - 1) * 2 * HP_MDT * 16 * (size_t)nprob;
}

// Largest cluster size C (16, 8 .. 1; at most one block per 16 rows) for which the nprob
// clusters of C blocks are all resident at once, as the occupancy calculator reports.  Where none is:
// the fewest blocks that a matrix's vectors fit in, beside x unless that takes more than twice as many
// as in x's space (fewer blocks leave fewer waves; with one or two more or less it is even).
// Stage `hetrd`, ms, x apart -> in vd's space: n = 2300, 16 problems (C = 7 -> 8) 529 -> 323, 64 problems (7 -> 3)
// 1471 -> 1174; n = 2500, 16 problems (16 -> 8) 620 -> 417, 64 problems (16 -> 4) 2106 -> 1224; n = 1250, 170
// problems (2 -> 1) 509 -> 583, which stays apart; n = 3000, 16 problems (FP64 form -> 8) 2131 -> 627.
int hetrd_mma_cluster_size(int n, int nprob, int num_sms, int digits) {
  const int NT = hd_tiles(n);
  const auto next = [](int c) { return c < 8 ? c + 1 : HP_MAX_CLUSTER; };
  int fit = 1, own = 1;
  while (fit < HP_MAX_CLUSTER && panel_form(n, fit).D == 0) fit = next(fit);
  while (own < HP_MAX_CLUSTER && (panel_form(n, own).D == 0 || panel_form(n, own).shared)) own = next(own);
  for (int c = HP_MAX_CLUSTER; c > fit; c = c > 8 ? 8 : c - 1) {
    if (c > NT || (long long)nprob * c > num_sms) continue;
    const PanelForm f = panel_form(n, c);
    const PanelFn fn = panel_fn(digits, f);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    int clusters = 0;
    if (panel_config(fn, cfg, attr, n, nprob, c, f, nullptr) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    if (clusters >= nprob) return c;
  }
  return own <= 2 * fit && !panel_form(n, own).shared ? own : fit;
}

cudaError_t launch_hetrd_panel_mma(int n, int nprob, const int32_t* size, z64* A, int ld, long long strideA, double* d,
                                   double* e, z64* tau, long long strideV, int i0, int C, const void* dig,
                                   const int* erow, int digits, void* md, z64* VWr, long long strideVW, cudaStream_t st) {
  const PanelForm f = panel_form(n, C);
  if ((digits != 6 && digits != HD_S) || f.D == 0) return cudaErrorInvalidValue;
  const PanelFn fn = panel_fn(digits, f);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  const cudaError_t err = panel_config(fn, cfg, attr, n, nprob, C, f, st);
  if (err != cudaSuccess) return err;
  return cudaLaunchKernelEx(&cfg, fn, n, size, A, ld, strideA, d, e, tau, strideV, i0, (const uint4*)dig, erow,
                            (uint4*)md, VWr, strideVW);
}

size_t hetrd_digits_bytes(int n, int nprob, int digits) {
  const size_t NT = hd_tiles(n);
  return NT * NT * 512 * (size_t)digits * (size_t)nprob;
}

cudaError_t launch_hetrd_digits(int n, int nprob, const int32_t* size, const z64* A, int ld, long long strideA, int i0,
                                void* dig, int* erow, int digits, cudaStream_t st) {
  const int L = n - i0 - 1;
  if (L <= 0) return cudaSuccess;
  dim3 grid((L + 15) / 16, nprob);
  if (digits == 6) hetrd_digits_kernel<6><<<grid, 256, 0, st>>>(n, size, A, ld, strideA, i0, (uint4*)dig, erow);
  else if (digits == HD_S) hetrd_digits_kernel<HD_S><<<grid, 256, 0, st>>>(n, size, A, ld, strideA, i0, (uint4*)dig, erow);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}
