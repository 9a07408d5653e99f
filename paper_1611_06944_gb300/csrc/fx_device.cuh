// Device helpers of the fixed-point format that dwf_fx.cuh describes.
#pragma once

#include "dwf_fx.cuh"

namespace hdcr {

typedef long long i64;
typedef unsigned long long u64;

constexpr int FX_UP = 5;  // a field's largest components: 2^57 <= |V| < 2^58; a link's one more

// V = 2^30 H + L, H the nearest integer
__device__ __forceinline__ int2 fx_limbs(i64 v) {
  const i64 t = v + (1LL << 29);
  return make_int2((int)(t >> 30), (int)((unsigned)t & 0x3fffffffu) - (1 << 29));
}

// V of one component of a group whose largest biased exponent is mx (in range), that exponent's
// numbers scaled to 2^(52 + up) .. 2^(53 + up), rounded to nearest
__device__ __forceinline__ i64 fx_fixed(double x, int mx, int up) {
  const int hi = __double2hiint(x);
  const int e = (hi >> 20) & 0x7ff;
  const int d = min(mx - e, 62);
  const u64 m = ((u64)(unsigned)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(x)) << up;
  const i64 v = (i64)((m + ((1ull << d) >> 1)) >> d);
  return hi < 0 ? -v : v;
}

// the largest biased exponent << 20 (and lower mantissa bits) of N complex numbers, and in bit
// 31 whether any is not zero
template <int N>
__device__ __forceinline__ unsigned fx_top(const cpx<double> (&x)[N]) {
  unsigned top = 0, any = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const unsigned a = __double2hiint(x[i].re) & 0x7fffffff, b = __double2hiint(x[i].im) & 0x7fffffff;
    top = max(top, max(a, b));
    any |= a | b | __double2loint(x[i].re) | __double2loint(x[i].im);
  }
  return top | (any != 0 ? 0x80000000u : 0u);
}

// the exponent mark of a group with that top
__device__ __forceinline__ int fx_mark(unsigned top, int emin, int emax) {
  const int mx = (int)(top >> 20) & 0x7ff;
  return !(top >> 31) ? 0 : mx < emin || mx > emax ? FX_RAW : mx;
}

// one number of a group with exponent mark ex (whose words are zero outside the format)
__device__ __forceinline__ int4 fx_encode(cpx<double> x, int ex, int up) {
  if (ex == 0 || ex == FX_RAW) return make_int4(0, 0, 0, 0);
  const int2 a = fx_limbs(fx_fixed(x.re, ex, up)), b = fx_limbs(fx_fixed(x.im, ex, up));
  return make_int4(a.x, a.y, b.x, b.y);
}

// r 2^(be - 1086), be the biased exponent that a leading bit 63 would have, rounded to nearest
__device__ __forceinline__ double fx_to_double(i64 r, int be) {
  const u64 m = (u64)(r < 0 ? -r : r);
  if (m == 0) return 0.0;
  const int lz = __clzll((i64)m);
  const u64 n = (m << lz) >> 1;  // leading bit 62
  const u64 q = ((n + 0x1ff + ((n >> 10) & 1)) >> 10) + ((u64)(be - lz - 1) << 52);
  return __longlong_as_double((i64)(q | ((u64)r & 0x8000000000000000ull)));
}

__device__ __forceinline__ i64 mw(int a, int b, i64 c) { return c + (i64)a * b; }

}  // namespace hdcr
