// Scalar parts of a Householder reflector shared by the reduction's kernels: square root and
// reciprocals by Newton's iteration.
#pragma once

#include "nao_internal.cuh"

__device__ __forceinline__ int hd_exp(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7ff); }

static __device__ __noinline__ double slow_sqrt(double q) { return sqrt(q); }
static __device__ __noinline__ double slow_reciprocal(double q) { return 1.0 / q; }

// sqrt(q) and 1 / sqrt(q) for q > 0 by Newton's iteration for the reciprocal root from a float
// seed, q scaled by an even power of two into [1, 4) (the library's sqrt and divisions take
// twice as many FP64 instructions, 64 cycles each in the one warp that forms a reflector)
__device__ __forceinline__ void sqrt_pair(double q, double& root, double& rroot) {
  const int b = hd_exp(q);
  if (b == 0 || b == 0x7ff) {
    root = slow_sqrt(q);
    rroot = slow_reciprocal(root);
    return;
  }
  const int k = (b - 1023) & ~1;
  const long long qb = __double_as_longlong(q) - ((long long)k << 52);
  const double m = __longlong_as_double(qb);
  // float bits of m: exponent 127 or 128, the top 23 mantissa bits
  const float f = __int_as_float((int)(((qb >> 52) - 1023 + 127) << 23) | (int)((qb >> 29) & 0x7fffff));
  const float yf = rsqrtf(f);
  const int yb = __float_as_int(yf);
  double y = __longlong_as_double((long long)((yb >> 23) - 127 + 1023) << 52 | (long long)(yb & 0x7fffff) << 29);
  const double h = 0.5 * m;
#pragma unroll
  for (int it = 0; it < 2; ++it) y = fma(y, fma(-h * y, y, 0.5), y);
  double g = m * y;
  g = fma(fma(-g, g, m), 0.5 * y, g);
  root = __longlong_as_double(__double_as_longlong(g) + ((long long)(k / 2) << 52));
  rroot = __longlong_as_double(__double_as_longlong(y) - ((long long)(k / 2) << 52));
}

// 1 / q for q > 0, in the same way
__device__ __forceinline__ double reciprocal(double q) {
  const int b = hd_exp(q);
  if (b < 3 || b > 2043) return slow_reciprocal(q);
  const long long qb = (__double_as_longlong(q) & 0xFFFFFFFFFFFFFll) | 1023ll << 52;
  const double m = __longlong_as_double(qb);
  const float f = __int_as_float(127 << 23 | (int)((qb >> 29) & 0x7fffff));
  const int yb = __float_as_int(__fdividef(1.0f, f));
  double y = __longlong_as_double((long long)((yb >> 23) - 127 + 1023) << 52 | (long long)(yb & 0x7fffff) << 29);
#pragma unroll
  for (int it = 0; it < 2; ++it) y = fma(y, fma(-m, y, 1.0), y);
  return __longlong_as_double(__double_as_longlong(y) - ((long long)(b - 1023) << 52));
}

// H = 1 - tau v v^H with v = (1, scale x(1:)) and H^H x = beta e_1, beta real, from alpha = x(0) and
// s = |x(1:)|^2; tau = 0 (H = 1) when there is nothing to eliminate
__device__ __forceinline__ void reflector(z64 alpha, double s, z64& tau, z64& scale, double& beta) {
  if (s == 0.0 && alpha.y == 0.0) {
    tau = zmk(0.0, 0.0);
    scale = zmk(0.0, 0.0);
    beta = alpha.x;
    return;
  }
  double root, rroot;
  sqrt_pair(fma(alpha.x, alpha.x, fma(alpha.y, alpha.y, s)), root, rroot);
  beta = -copysign(root, alpha.x);
  const double rb = -copysign(rroot, alpha.x);  // 1 / beta
  tau = zmk((beta - alpha.x) * rb, -alpha.y * rb);
  const z64 den = zmk(alpha.x - beta, alpha.y);  // scale = 1 / (alpha - beta)
  const double rd = reciprocal(zabs2(den));
  scale = zmk(den.x * rd, -den.y * rd);
}
