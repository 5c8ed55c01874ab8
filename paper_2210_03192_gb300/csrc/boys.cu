// Host construction of the Boys-function interpolation tables used by the
// integral kernels (paper Sec. 2.5.2: 7th-order Chebyshev interpolation on
// intervals, upward recursion in m beyond x = 117).
//
// Design on GB300: the kernels evaluate only the highest order F_L(T) and
// exp(-T) from the table (two degree-7 polynomials) and obtain F_m for
// m = L-1 .. lc by the downward relation (2m+1) F_m = 2T F_{m+1} + exp(-T),
// which is stable.  For T >= 117 exp(-T) is negligible next to every
// F_m (m <= 24) in FP64 and F_L = Gamma(L+1/2)/2 * T^{-(L+1/2)} exactly to
// FP64, so the same downward relation with exp(-T) = 0 applies.  That range
// is tabulated too, on 256 intervals per octave up to 2^24: one FP64
// instruction costs 64 issue slots, and a separate asymptotic branch (a root,
// a reciprocal and powers, 16 instructions) was paid by nearly every warp,
// whose kets lie on both sides of 117.
//
// Reference values for the fit: F_m(T) = exp(-T) sum_i (2T)^i /
// ((2m+1)(2m+3)...(2m+2i+1)), a series of positive terms, summed in long double.
#include <cmath>

#include "lx3c_internal.h"

namespace lx3c {

long double boys_ref(int m, long double T) {
  long double term = 1.0L / (2 * m + 1), sum = term;
  for (int i = 1; i < 20000; ++i) {
    term *= 2.0L * T / (long double)(2 * m + 2 * i + 1);
    sum += term;
    if (term < 1e-30L * sum) break;
  }
  return std::exp(-T) * sum;
}

double boys_large_const(int L) {
  // Gamma(L + 1/2) / 2 = (2L-1)!! / 2^{L+1} * sqrt(pi)
  long double g = std::sqrt(3.14159265358979323846264338327950288L);
  for (int k = 1; k <= L; ++k) g *= (k - 0.5L);
  return (double)(g / 2.0L);
}

namespace {

// Monomial coefficients, in powers of T - c, of the Chebyshev interpolant of a
// function given by its values fk at the nodes c + h cos(pi (k + 1/2) / n).
struct ChebFit {
  static constexpr int n = kBoysDeg + 1;
  long double x[n], cs[n][n], mono[n][n];  // nodes; T_j at the nodes; T_j in monomials
  ChebFit() {
    const long double pi = 3.14159265358979323846264338327950288L;
    for (int k = 0; k < n; ++k) x[k] = std::cos(pi * (k + 0.5L) / n);
    for (int j = 0; j < n; ++j)
      for (int k = 0; k < n; ++k) {
        cs[j][k] = std::cos(pi * j * (k + 0.5L) / n);
        mono[j][k] = 0;
      }
    mono[0][0] = 1;
    mono[1][1] = 1;
    for (int j = 2; j < n; ++j)
      for (int k = 0; k < n; ++k) mono[j][k] = -mono[j - 2][k] + (k > 0 ? 2 * mono[j - 1][k - 1] : 0);
  }
  void operator()(const long double* fk, long double h, double* out) const {
    long double m[n] = {0};
    for (int j = 0; j < n; ++j) {
      long double s = 0;
      for (int k = 0; k < n; ++k) s += fk[k] * cs[j][k];
      s *= (j ? 2.0L : 1.0L) / n;
      for (int k = 0; k <= j; ++k) m[k] += s * mono[j][k];
    }
    long double sc = 1;
    for (int k = 0; k < n; ++k) {
      out[k] = (double)(m[k] / sc);
      sc *= h;
    }
  }
};

}  // namespace

// tab[(i*kBoysNF + f)*8 + j]: coefficient of (T - mid_i)^j for function f
// (f <= kBoysMmax: F_f, f = kBoysMmax+1: exp(-T)) on interval i; intervals of
// width 1/8 up to 117, then those of kBoysOct per octave.
void boys_tables(std::vector<double>& tab, std::vector<double>& mid) {
  const ChebFit fit;
  const int n = ChebFit::n;
  tab.assign((size_t)kBoysNInt * kBoysNF * 8, 0.0);
  mid.assign(kBoysNInt, 0.0);
  const long double h = 0.5L / kBoysPerUnit;  // half width
  for (int i = 0; i < kBoysNLin; ++i) {
    const long double c = (i + 0.5L) / kBoysPerUnit;
    mid[i] = (double)c;
    for (int f = 0; f < kBoysNF; ++f) {
      long double fk[n];
      for (int k = 0; k < n; ++k) fk[k] = (f <= kBoysMmax) ? boys_ref(f, c + h * fit.x[k]) : std::exp(-(c + h * fit.x[k]));
      fit(fk, h, &tab[((size_t)i * kBoysNF + f) * 8]);
    }
  }
  // T >= 117: F_f(4 T) = F_f(T) 2^{-(2f+1)}, so two octaves give all
  const long double spi = std::sqrt(3.14159265358979323846264338327950288L);
  std::vector<double> base((size_t)2 * kBoysOct * (kBoysMmax + 1) * 8);
  for (int j = 0; j < 2 * kBoysOct; ++j) {
    const long double w = j < kBoysOct ? 64.0L / kBoysOct : 128.0L / kBoysOct;
    const long double c = (j < kBoysOct ? 64.0L : 128.0L) + (j % kBoysOct + 0.5L) * w;
    long double F[kBoysMmax + 1][n];
    for (int k = 0; k < n; ++k) {
      const long double T = c + 0.5L * w * fit.x[k];
      long double v = 0.5L * spi / std::sqrt(T);
      for (int f = 0; f <= kBoysMmax; ++f) {
        F[f][k] = v;
        v *= (f + 0.5L) / T;
      }
    }
    for (int f = 0; f <= kBoysMmax; ++f) fit(F[f], 0.5L * w, &base[((size_t)j * (kBoysMmax + 1) + f) * 8]);
  }
  for (int i = kBoysNLin; i < kBoysNInt; ++i) {
    const int j = i - kBoysNLin + kBoysOctFirst, oct = j / kBoysOct, s = oct & ~1;  // T = 2^s x base T
    const int bj = (oct & 1) * kBoysOct + j % kBoysOct;
    mid[i] = std::ldexp((64.0 + (j % kBoysOct + 0.5) * (64.0 / kBoysOct)), oct);
    for (int f = 0; f <= kBoysMmax; ++f)
      for (int k = 0; k < n; ++k)
        tab[((size_t)i * kBoysNF + f) * 8 + k] =
            std::ldexp(base[((size_t)bj * (kBoysMmax + 1) + f) * 8 + k], -(s * (f + k) + s / 2));
  }
}

}  // namespace lx3c
