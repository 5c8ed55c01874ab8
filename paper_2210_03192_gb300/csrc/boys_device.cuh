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

// 1/sqrt(x) for x > 0 in FP64: single-precision seed, then one Newton-Raphson
// step carrying the second-order term (y1 = y0 (1 + e/2 + 3e^2/8),
// e = 1 - x y0^2), which takes the ~1e-7 seed error to FP64 rounding level
// with five FP64 operations.
__device__ __forceinline__ double rsqrt_fp64(double x) {
  float xf = __double2float_rn(x);
  double y0 = (double)rsqrtf(xf);
  double t = x * y0;
  double e = fma(-t, y0, 1.0);
  double p = fma(e, 0.375, 0.5);
  double q = y0 * e;
  return fma(q, p, y0);
}

// F_hi(T) and, when want_ex, exp(-T) for the downward relation: interpolation
// table for T < 117, else the asymptotic form with exp(-T) = 0.
__device__ __forceinline__ void boys_top(const double* __restrict__ tab, const double* __restrict__ mid, double cL,
                                         int hi, bool want_ex, double T, double& FL, double& ex) {
  ex = 0.0;
  if (T < kBoysTMax) {
    int i = __float2int_rz(__double2float_rz(T) * (float)kBoysPerUnit);
    i = min(max(i, 0), kBoysNInt - 1);
    const double dx = T - __ldg(mid + i);
    const double* c = tab + ((size_t)i * kBoysNF + hi) * 8;
    const double* ce = tab + ((size_t)i * kBoysNF + (kBoysNF - 1)) * 8;
    FL = __ldg(c + 7);
    if (want_ex) {
      ex = __ldg(ce + 7);
#pragma unroll
      for (int j = 6; j >= 0; --j) {
        FL = fma(FL, dx, __ldg(c + j));
        ex = fma(ex, dx, __ldg(ce + j));
      }
    } else {
#pragma unroll
      for (int j = 6; j >= 0; --j) FL = fma(FL, dx, __ldg(c + j));
    }
  } else {
    const double rs = rsqrt_fp64(T);
    // 1/T from the root, one Newton step (a fresh reciprocal costs twice the
    // instructions, and most warps hold lanes on both sides of 117)
    double b = rs * rs;
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
