// Device arithmetic shared by the integral kernels: FP64 reciprocal roots from
// FP32 seeds and the Boys function (Sec. 2.5.2).
#pragma once
#include <cuda_runtime.h>

#include "lx3c_internal.h"

namespace lx3c {

// 1/n, n = 1..47 (entry 0 unused)
static __constant__ double c_inv[48] = {
    0.0,      1.0,      1.0 / 2,  1.0 / 3,  1.0 / 4,  1.0 / 5,  1.0 / 6,  1.0 / 7,  1.0 / 8,  1.0 / 9,
    1.0 / 10, 1.0 / 11, 1.0 / 12, 1.0 / 13, 1.0 / 14, 1.0 / 15, 1.0 / 16, 1.0 / 17, 1.0 / 18, 1.0 / 19,
    1.0 / 20, 1.0 / 21, 1.0 / 22, 1.0 / 23, 1.0 / 24, 1.0 / 25, 1.0 / 26, 1.0 / 27, 1.0 / 28, 1.0 / 29,
    1.0 / 30, 1.0 / 31, 1.0 / 32, 1.0 / 33, 1.0 / 34, 1.0 / 35, 1.0 / 36, 1.0 / 37, 1.0 / 38, 1.0 / 39,
    1.0 / 40, 1.0 / 41, 1.0 / 42, 1.0 / 43, 1.0 / 44, 1.0 / 45, 1.0 / 46, 1.0 / 47};

// FP64 <-> FP32 by shifting bits: the conversion instructions run at the FP64
// rate (17 SM clocks per warp, measured), these in the integer pipe.  Values
// from 2^128 on give infinity, those below 2^-127 zero (high word clamped, low
// word cleared).
__device__ __forceinline__ float to_float_bits(double x) {  // x >= 0, truncated
  const int h = __double2hiint(x), hi = min(max(h, 0x38000000), 0x47F00000);
  const unsigned lo = h == hi ? (unsigned)__double2loint(x) : 0u;
  return __int_as_float((int)__funnelshift_l(lo, (unsigned)(hi - 0x38000000), 3));
}
__device__ __forceinline__ double to_double_bits(float y) {  // finite y > 0, or 0
  const int b = __float_as_int(y);
  return __hiloint2double(b ? (b >> 3) + 0x38000000 : 0, b << 29);
}

// 1/sqrt(x) in FP64 for x in the range of a normal float: single-precision
// seed, then one Newton-Raphson step carrying the second-order term
// (y1 = y0 (1 + e/2 + 3e^2/8), e = 1 - x y0^2), which takes the ~1e-7 seed
// error to FP64 rounding level with five FP64 operations.  0 from 2^128 on.
__device__ __forceinline__ double rsqrt_fp64(double x) {
  double y0 = to_double_bits(rsqrtf(to_float_bits(x)));
  double t = x * y0;
  double e = fma(-t, y0, 1.0);
  double p = fma(e, 0.375, 0.5);
  double q = y0 * e;
  return fma(q, p, y0);
}

// F_hi(T) and, when want_ex, exp(-T) for the downward relation, by degree-7
// interpolation: the interval from the bits of T (floor(8 T) below 117, the
// top mantissa bits up to 2^24), the asymptotic form with exp(-T) = 0 beyond.
__device__ __forceinline__ void boys_top(const double* __restrict__ tab, const double* __restrict__ mid, double cL,
                                         int hi, bool want_ex, double T, double& FL, double& ex) {
  constexpr int kHi117 = 0x405D4000, kHi24 = 0x41700000;  // high words of 117 and 2^24
  const int h = __double2hiint(T);
  ex = 0.0;
  if (h < kHi24) {
    const int lin = ((h & 0xFFFFF) | 0x100000) >> min(1040 - (h >> 20), 31);
    const int i = h < kHi117 ? lin : kBoysNLin + ((h >> 12) - (kHi117 >> 12));
    const double dx = T - __ldg(mid + i);
    const double2* c = reinterpret_cast<const double2*>(tab + ((size_t)i * kBoysNF + hi) * 8);
    const double2* ce = reinterpret_cast<const double2*>(tab + ((size_t)i * kBoysNF + (kBoysNF - 1)) * 8);
    const double2 c0 = __ldg(c), c1 = __ldg(c + 1), c2 = __ldg(c + 2), c3 = __ldg(c + 3);
    FL = fma(fma(fma(fma(fma(fma(fma(c3.y, dx, c3.x), dx, c2.y), dx, c2.x), dx, c1.y), dx, c1.x), dx, c0.y), dx, c0.x);
    if (want_ex) {
      const double2 e0 = __ldg(ce), e1 = __ldg(ce + 1), e2 = __ldg(ce + 2), e3 = __ldg(ce + 3);
      ex = fma(fma(fma(fma(fma(fma(fma(e3.y, dx, e3.x), dx, e2.y), dx, e2.x), dx, e1.y), dx, e1.x), dx, e0.y), dx, e0.x);
    }
  } else {
    // the root of T 4^-k in [1, 4), for any finite T (NaN and infinity give NaN)
    const int k = h < 0x7FF00000 ? ((h >> 20) - 1023) >> 1 : 0;
    const double rs = rsqrt_fp64(__hiloint2double(h - (k << 21), __double2loint(T))) *
                      __hiloint2double((1023 - k) << 20, 0);
    double b = rs * rs;  // 1/T, one Newton step from the root
    b = fma(b, fma(-T, b, 1.0), b);
    double p = rs;
    int e = hi;
    while (e) {
      if (e & 1) p *= b;
      e >>= 1;
      if (e) b *= b;
    }
    FL = cL * p;
  }
}

}  // namespace lx3c
