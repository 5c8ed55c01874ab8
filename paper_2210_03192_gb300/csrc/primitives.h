// Which primitive pairs of a shell pair contribute to its integrals (host and
// device: the planners and the allocation-free path's orientation kernel).
#pragma once
#include <cmath>

namespace lx3c {

// A primitive pair whose Schwarz bound is below kPrimDrop of the shell pair's
// largest is left out: its share of any integral, at most that fraction of
// the bound of the block, is 14 orders below FP64 rounding of the block's
// elements.  Half the primitive pairs of a contracted shell pair a few bohr
// apart fall under it (their Gaussian product exp(-za zb/(za+zb) R^2) is
// 1e-40 or, in most of these cases, 0 in FP64): measured on shells with
// exponents in [0.05, 1e4], K = 6, in a 20-bohr box, 35 % remain, of the
// 61 % with a nonzero product.
constexpr double kPrimDrop = 1e-30;

// K: the pair's prefactor c_a c_b exp(-za zb/gamma R^2), zero when the
// Gaussian product underflows (the pair then contributes exactly nothing).
// Returns the bound: sqrt of the (ss|ss) self-repulsion times the rms size of
// (x-A)^la (x-B)^lb under the product, up to a common factor.
__host__ __device__ inline double prim_bound(double za, double ca, double zb, double cb, double ab2, int la, int lb,
                                             double* K) {
  const double g = za + zb, ig = 1.0 / g;
  *K = ca * cb * exp(-za * zb * ig * ab2);
  const double ra = sqrt(zb * ig * zb * ig * ab2 + 0.5 * ig), rb = sqrt(za * ig * za * ig * ab2 + 0.5 * ig);
  double q = fabs(*K) * ig * sqrt(sqrt(ig));
  for (int i = 0; i < la; ++i) q *= ra;
  for (int i = 0; i < lb; ++i) q *= rb;
  return q;
}

__host__ __device__ inline bool prim_kept(double K, double q, double qmax) {
  return K != 0.0 && !(q < kPrimDrop * qmax);
}

}  // namespace lx3c
