// The Hermite DF-J kernel (hermite.cu has the mathematics) for the classes
// that carry most of a build, Hermite degree up to 6, with every sum written out
// at compile time and its operands in registers.
//
// With
//   M_n = R^n / n!,  Z_u = sum_e H~_{u+e} R~_e,  X_u = sum_c CP_{u+c} M_c / u!
// the polynomial shifts are two short convolutions,
//   G_c += sum_u Z_u / u! M_{c-u},   y_a = sum_{u <= a} R~_{a-u} X_u
// (G_c: gamma in Cartesian monomials over c!, |c| = lc; CP_c the ket's q).
// For these degrees that is fewer operations than the axis-by-axis shifts
// ((pp|g): 81 terms instead of 109 for gamma), and none of the table words,
// operand loads and column stores that held the table kernel to 62 to 78 % of
// the FP64 pipe.  R, M and G live in registers (up to 255, eight one-warp
// blocks per SM, two per sub-partition: FP64 latency equals its issue
// interval, so two suffice); CP, X and the densities in shared memory.
// Where R, M and G together pass 255 registers (degree 5 and 6, ket l = 6), M
// is read from shared memory.  Spills (stores / loads, the worst class of a
// kernel): degree 4 340 / 376 B, 5 636 / 680 B, 6 3.1 / 3.6 KB; degree 7 on,
// whose R alone is 240 registers, stays with the table kernel.  Against the table
// kernel: DF-J of 32 atoms 103.2 -> 71.1 ms (degrees 2 to 4 alone 80.4), a
// batch of three molecules 11.9 -> 8.9 ms, energy and gradient of 12 atoms
// 29.6 -> 25.4 ms.
#pragma once
#include <utility>

#include "boys_device.cuh"
#include "hermite_device.cuh"

namespace lx3c {

namespace {

// f(0), f(1), ... with constant arguments
template <int I>
struct Const {
  __host__ __device__ constexpr operator int() const { return I; }
};
template <class F, int... I>
__device__ __forceinline__ void each_of(std::integer_sequence<int, I...>, const F& f) {
  (f(Const<I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void each(const F& f) {
  each_of(std::make_integer_sequence<int, N>{}, f);
}

struct Mono {
  int x, y, z;
};
// exponents of graded index h
__host__ __device__ constexpr Mono mono(int h) {
  int n = 0;
  while (nherm(n) <= h) ++n;
  const int r = h - nherm(n - 1);
  int m = 0;
  while ((m + 1) * (m + 2) / 2 <= r) ++m;
  const int z = r - m * (m + 1) / 2;
  return Mono{n - m, m - z, z};
}
// on graded indices: degree, sum, difference, order, product of factorials
__host__ __device__ constexpr int deg(int a) { return mono(a).x + mono(a).y + mono(a).z; }
__host__ __device__ constexpr int add(int a, int b) {
  return hidx(mono(a).x + mono(b).x, mono(a).y + mono(b).y, mono(a).z + mono(b).z);
}
__host__ __device__ constexpr int sub(int a, int b) {
  return hidx(mono(a).x - mono(b).x, mono(a).y - mono(b).y, mono(a).z - mono(b).z);
}
__host__ __device__ constexpr bool le(int a, int b) {
  return mono(a).x <= mono(b).x && mono(a).y <= mono(b).y && mono(a).z <= mono(b).z;
}
__host__ __device__ constexpr double fact3(int a) {
  double f = 1.0;
  for (int i = 2; i <= mono(a).x; ++i) f *= i;
  for (int i = 2; i <= mono(a).y; ++i) f *= i;
  for (int i = 2; i <= mono(a).z; ++i) f *= i;
  return f;
}
// axis of the smallest nonzero exponent, that exponent, and k steps down it
__host__ __device__ constexpr int axis(int a) {
  const Mono m = mono(a);
  int best = -1, n = 1000;
  if (m.x > 0 && m.x < n) { best = 0; n = m.x; }
  if (m.y > 0 && m.y < n) { best = 1; n = m.y; }
  if (m.z > 0 && m.z < n) { best = 2; n = m.z; }
  return best;
}
__host__ __device__ constexpr int power(int a) {
  return axis(a) == 0 ? mono(a).x : (axis(a) == 1 ? mono(a).y : mono(a).z);
}
__host__ __device__ constexpr int down(int a, int k) {
  const Mono m = mono(a);
  return hidx(m.x - (axis(a) == 0 ? k : 0), m.y - (axis(a) == 1 ? k : 0), m.z - (axis(a) == 2 ? k : 0));
}

constexpr int least(int a, int b) { return a < b ? a : b; }
constexpr int kRowsMost = 32;  // y rows staged at a time

template <int Lab, int LC>
struct Shape {
  static constexpr int NR = nherm(Lab), NCC = (LC + 1) * (LC + 2) / 2, KU = least(Lab, LC), NU = nherm(KU),
                       NM = nherm(LC), C0 = nherm(LC - 1), NROW = least(NR, kRowsMost),
                       M0 = nherm(LC - KU - 1);  // the first monomial in use
  // M in shared memory where R, M and G together pass 255 registers; the rows
  // of y are staged over it, and the next ket primitive forms it again
  static constexpr bool kMShared = unrolled_m_shared(Lab, LC);
};

template <int Lab, int LC>
__device__ __forceinline__ void herm_tile(const HermArgs& g, const HermCls& c, const int4& tile, int mode, double* sm) {
  using S = Shape<Lab, LC>;
  constexpr int NR = S::NR, NCC = S::NCC, NU = S::NU;
  const int lane = threadIdx.x;
  const int W = c.W, NP = 32 / W, grp = lane / W;
  const int q = tile.y + (lane - grp * W);
  const int qc = min(q, c.nket - 1);
  double* Hs = sm;
  double* CP = sm + (NP * NR + 31) / 32 * 32 + lane;  // columns: CP, then X
  double* X = CP + NCC * 32;
  double* stg = X - lane + NU * 32;
  double* MS = stg + lane;
  const double Cx = __ldg(c.auxc + 3 * qc), Cy = __ldg(c.auxc + 3 * qc + 1), Cz = __ldg(c.auxc + 3 * qc + 2);
  const int ao = __ldg(c.aux_ao + qc);
  double f0 = 0.0, f1 = 0.0, f2 = 0.0;
  double G[NCC];
  each<NCC>([&](auto n) { G[n] = 0.0; });
  if (mode & 6) {
    for (int n = 0; n < NCC; ++n) {
      double v = 0.0;
      for (int k = __ldg(c.cptr + n); k < __ldg(c.cptr + n + 1); ++k) {
        const int2 e = __ldg(c.cent + k);
        v = fma(__ldg(c.pal + e.y), __ldg(g.cvec + ao + e.x), v);
      }
      CP[n * 32] = v;
    }
  }
  for (int e0 = 0; e0 < tile.w; e0 += NP) {
    const int ie = e0 + grp;
    const int prim = tile.z + min(ie, tile.w - 1);
    const bool act = ie < tile.w && q < __ldg(c.cnt + __ldg(c.primpair + prim));
    const double* pr = c.prim + 4LL * prim;
    const double gam = __ldg(pr);
    const double R3[3] = {__ldg(pr + 1) - Cx, __ldg(pr + 2) - Cy, __ldg(pr + 3) - Cz};
    const double R2 = fma(R3[2], R3[2], fma(R3[1], R3[1], R3[0] * R3[0]));
    if (mode & 1) {
      // the densities of the NP primitive pairs, side by side
      __syncwarp();
      for (int s = 0; s < NP; ++s) {
        const double* H = c.H + (long long)(tile.z + min(e0 + s, tile.w - 1)) * NR;
        for (int t = lane; t < NR; t += 32) Hs[s * NR + t] = __ldg(H + t);
      }
      __syncwarp();
    }
    const double* Hg = Hs + grp * NR;
    double M[S::NM];
    const auto monomials = [&]() {
      each<S::NM>([&](auto i) {
        constexpr int h = i;
        if constexpr (h == 0) M[h] = 1.0;
        else if constexpr (deg(h) == 1) M[h] = R3[axis(h)];
        else if constexpr (power(h) == 1) M[h] = R3[axis(h)] * M[down(h, 1)];
        else M[h] = (R3[axis(h)] * (1.0 / power(h))) * M[down(h, 1)];
        if constexpr (S::kMShared && h >= S::M0) MS[(h - S::M0) * 32] = M[h];
      });
    };
    const auto mono_at = [&](auto i) {
      constexpr int h = i;
      if constexpr (S::kMShared) return MS[(h - S::M0) * 32];
      else return M[h];
    };
    monomials();
    if (mode & 6)
      each<NU>([&](auto i) {
        constexpr int u = i, n = LC - deg(u), w0 = nherm(n - 1);
        double x = 0.0;
        each<nherm(n) - w0>([&](auto j) {
          constexpr int w = w0 + j;
          const double cp = CP[(add(u, w) - S::C0) * 32];
          const double mw = mono_at(Const<w>{});
          x = w == w0 ? cp * mw : fma(cp, mw, x);
        });
        if constexpr (fact3(u) != 1.0) x *= 1.0 / fact3(u);
        X[u * 32] = x;
      });
#pragma unroll 1
    for (int ic = 0; ic < c.Kc; ++ic) {
      if (S::kMShared && ic > 0 && (mode & 1)) monomials();
      const double zc = __ldg(c.auxrec + ((long long)qc * c.Kc + ic) * kAuxRec);
      const double ccp = __ldg(c.auxrec + ((long long)qc * c.Kc + ic) * kAuxRec + 1);
      const double rs = rsqrt_fp64(gam + zc);
      const double r = rs * rs;
      const double gr = gam * r;
      const double rho = gr * zc;
      const double n2r = -2.0 * rho;
      double pref = ccp * rs;
      {
        double b = gr;
#pragma unroll
        for (int e = LC; e; e >>= 1) {
          if (e & 1) pref *= b;
          if (e > 1) b *= b;
        }
      }
      if (!act) pref = 0.0;
      double FL, ex;
      boys_top(g.boys_tab, g.boys_mid, c.boys_cL, Lab + LC, true, rho * R2, FL, ex);
      double fm = pref * FL;
      double B[Lab];
      {
        double b = n2r;
#pragma unroll
        for (int e = Lab; e; e >>= 1) {
          if (e & 1) fm *= b;
          if (e > 1) b *= b;
        }
        B[0] = pref * ex;
#pragma unroll
        for (int m = 1; m < Lab; ++m) B[m] = B[m - 1] * n2r;
      }
      // R~_e^(m) = (X R~_{e-1}^(m+1) + R~_{e-2}^(m+1)) / e_axis, degrees
      // descending in place
      double R[NR];
      R[0] = fm;
      each<Lab>([&](auto step) {
        constexpr int m = Lab - 1 - step, top = nherm(Lab - m);
        each<top - 1>([&](auto k) {
          constexpr int h = top - 1 - k;
          if constexpr (power(h) == 1) R[h] = R3[axis(h)] * R[down(h, 1)];
          else R[h] = fma(R3[axis(h)], R[down(h, 1)], R[down(h, 2)]) * (1.0 / power(h));
        });
        fm = fma(-R2, fm, B[m]) * (1.0 / (2 * (LC + m) + 1));
        R[0] = fm;
      });
      if (mode & 1)
        each<NU>([&](auto i) {
          constexpr int u = i, n = LC - deg(u), w0 = nherm(n - 1);
          double z = Hg[u] * R[0];
          each<nherm(Lab - deg(u)) - 1>([&](auto j) {
            constexpr int e = j + 1;
            z = fma(Hg[add(u, e)], R[e], z);
          });
          if constexpr (fact3(u) != 1.0) z *= 1.0 / fact3(u);
          each<nherm(n) - w0>([&](auto j) {
            constexpr int w = w0 + j, cc = add(u, w) - S::C0;
            G[cc] = fma(z, mono_at(Const<w>{}), G[cc]);
          });
        });
      if (mode & 6) {
        if (S::kMShared) __syncwarp();  // rows go over the other lanes' M
        const double* Hf = c.H + 3LL * prim * NR;  // gradient
        each<NR>([&](auto i) {
          constexpr int a = i;
          double y = R[a] * X[0];
          each<NU - 1>([&](auto j) {
            constexpr int u = j + 1;
            if constexpr (le(u, a)) y = fma(R[sub(a, u)], X[u * 32], y);
          });
          constexpr int row = a % S::NROW;
          stg[row * 33 + lane] = y;
          if (mode & 4) {
            if constexpr (mono(a).x > 0) f0 = fma(__ldg(Hf + a), y, f0);
            if constexpr (mono(a).y > 0) f1 = fma(__ldg(Hf + NR + a), y, f1);
            if constexpr (mono(a).z > 0) f2 = fma(__ldg(Hf + 2 * NR + a), y, f2);
          }
          if constexpr (row == S::NROW - 1 || a == NR - 1)
            sum_rows(c, stg, row + 1, tile, e0, lane, [&](int r) { return a - row + r; });
        });
      }
    }
  }
  if (mode & 1) {
    each<NCC>([&](auto n) { CP[n * 32] = G[n]; });
    if (q < c.nket)
      for (int C = 0; C < 2 * LC + 1; ++C) {
        double v = 0.0;
        for (int k = __ldg(c.gptr + C); k < __ldg(c.gptr + C + 1); ++k) {
          const int2 e = __ldg(c.gent + k);
          v = fma(__ldg(c.pal + e.y), CP[e.x * 32], v);
        }
        fix_add(g.gacc + kFixWords * (ao + C), v);
      }
  }
  if ((mode & 4) && q < c.nket) {
    unsigned long long* f = g.facc + kFixWords * 3 * (long long)__ldg(c.aux_atom + qc);
    fix_add(f, -f0);
    fix_add(f + kFixWords, -f1);
    fix_add(f + 2 * kFixWords, -f2);
  }
}

template <int Lab>
__global__ void __launch_bounds__(32, 8) herm_unrolled_kernel(const __grid_constant__ HermArgs g, int mode) {
  extern __shared__ double sm[];
  const int4 tile = __ldg(g.tiles + blockIdx.x);
  const HermCls& c = g.cls[tile.x];
  each<7>([&](auto i) {
    if constexpr (herm_unrolled(Lab, i))
      if (c.lc == i) herm_tile<Lab, i>(g, c, tile, mode, sm);
  });
}

}  // namespace

// The kernel of one Lab: setup allows it the shared memory, a launch runs n
// tiles.
#define LX3C_HERM_UNROLLED(LAB)                                                                              \
  template <>                                                                                                \
  cudaError_t herm_unrolled_setup<LAB>() {                                                                   \
    return cudaFuncSetAttribute(herm_unrolled_kernel<LAB>, cudaFuncAttributeMaxDynamicSharedMemorySize, 65536); \
  }                                                                                                          \
  template <>                                                                                                \
  cudaError_t herm_unrolled_launch<LAB>(const HermArgs& a, int mode, int smem, long long n, cudaStream_t st) { \
    herm_unrolled_kernel<LAB><<<(unsigned)n, 32, smem, st>>>(a, mode);                                       \
    return cudaGetLastError();                                                                               \
  }

}  // namespace lx3c
