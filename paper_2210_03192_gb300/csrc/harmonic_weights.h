// The ket's harmonic weights W_{k,m} = Y^k s_{lc-k,m}(X) (plan.cu has the
// scheme), formed for one |m| at a time: the integral kernels' weight stage,
// and the host evaluation of the class tables.
#pragma once

namespace lx3c {

// (l^2 - m^2) / (4 l^2 - 1), l, m <= 5, of the recursion
// Q_{l+1,m} = z Q_{l,m} - c r^2 Q_{l-1,m}, at [6 l + m]
#define LX3C_QC(l, m) ((double)((l) * (l) - (m) * (m)) / (4.0 * (l) * (l) - 1.0))
#define LX3C_QROW(l) \
  LX3C_QC(l, 0), LX3C_QC(l, 1), LX3C_QC(l, 2), LX3C_QC(l, 3), LX3C_QC(l, 4), LX3C_QC(l, 5)
#define LX3C_QTABLE \
  { 0, 0, 0, 0, 0, 0, LX3C_QROW(1), LX3C_QROW(2), LX3C_QROW(3), LX3C_QROW(4), LX3C_QROW(5) }

// lc > 0.  (x + i y)^m, then Q_{l,m}(z, r^2) for l = m..lc; q: the table above,
// yk(k) = Y^k, put(index, value) takes W_{k,m} and W_{k,-m} for k <= kmax.
template <class Q, class Yk, class Put>
__host__ __device__ __forceinline__ void harmonic_weights(int lc, int kmax, int m, double X, double Yc, double Z,
                                                          const Q& q, const Yk& yk, const Put& put) {
  const double r2 = fma(Z, Z, fma(Yc, Yc, X * X));
  double A = X, B = Yc;
  for (int i = 1; i < m; ++i) {
    const double An = fma(A, X, -B * Yc);
    B = fma(A, Yc, B * X);
    A = An;
  }
  double q0 = 0.0, q1 = 1.0;
  for (int l = m; l <= lc; ++l) {
    const int k = lc - l;
    if (k <= kmax) {
      const double v = k ? q1 * yk(k) : q1;
      const int o = k * (2 * lc + 2 - k) + l;  // m = 0 of degree l
      if (m == 0) {
        put(o, v);
      } else {
        put(o + m, v * A);
        put(o - m, v * B);
      }
    }
    if (l < lc) {
      double n = Z * q1;
      if (l > m) n = fma(-q[l * 6 + m] * r2, q0, n);
      q0 = q1;
      q1 = n;
    }
  }
}

}  // namespace lx3c
