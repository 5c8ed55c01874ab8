// DF-J build and gradient in a Hermite Gaussian basis (the J-engine the paper
// names as follow-up work, Sec. 4).  The density of a primitive pair is
// expanded once per pair in Hermite Gaussians Lambda_a, |a| <= la + lb
// (McMurchie-Davidson), and each primitive triple then needs only
//   (Lambda_a|C) = d_P^a [ S_C(R) f(R^2) ],   R = P - C,
// with the solid-harmonic ket in closed form (Hobson: S_C(d) F_0 =
// S_C(R) (-2 rho)^lc F_lc).  By Leibniz' rule, with
//   R_e = d^e [pref F_lc(rho R^2)]  (Hermite integrals of base order lc),
//   q   = sum_C c_C S_C             (a polynomial of degree lc),
// the two contractions are polynomial products,
//   gamma_C = sum_u d^u S_C(R) / u! Z_u,   Z_u = sum_e H~_{u+e} R~_e,
//   y_a/a!  = sum_{u <= a} R~_{a-u} (d^u q(R) / u!),   J_ab = sum_a E^ab_a y_a,
// (H~_a = a! H_a, R~_e = R_e/e!, u <= lc), and d^u S_C(R), d^u q(R) are Taylor
// shifts of the Cartesian polynomials, one axis at a time.  No integral (ab|C)
// is formed: (ff|h) costs about 2.8e3 FP64 instructions per triple where
// forming and digesting its integrals took 3.4e4 flops.
//
// The classes of degree up to 6 run on the unrolled kernel of
// hermite_unrolled.cuh; this file has the tables and the kernel for the others,
// the kernels per pair, and the plans of both.
//
// GB300 layout.  FP64 issues one warp instruction per 16 SM clocks, so an FMA
// may spend 16 clocks of shared-memory bandwidth and 64 issue slots on its
// operands: every stage runs from per-lane shared-memory columns driven by
// small index tables, with all 32 lanes on one table entry.  A block owns a
// tile (W kets x a range of primitive pairs, 32/W pairs at a time); a lane
// reads and writes only its own columns, so a one-warp block needs no barrier
// and no lane idles beyond the ragged end of a ket list.  An SM sub-partition
// issues one FP64 warp instruction per 64 clocks, so it takes eight or more
// warps to keep the four busy: where the columns of a class let fewer one-warp
// blocks onto an SM, two or four warps share the columns and divide every
// stage's outputs, with a barrier between stages.
#include <algorithm>
#include <array>
#include <cmath>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <tuple>

#include "../../include/lx3c.h"
#include "boys_device.cuh"
#include "fixed128.cuh"
#include "hermite.h"
#include "hermite_device.cuh"
#include "primitives.h"

namespace lx3c {

namespace {

__constant__ double c_int[16] = {0., 1., 2., 3., 4., 5., 6., 7., 8., 9., 10., 11., 12., 13., 14., 15.};

__device__ __forceinline__ double lds(const char* base, unsigned off) { return *(const double*)(base + off); }
__device__ __forceinline__ void sts(char* base, unsigned off, double v) { *(double*)(base + off) = v; }

// Runs a stage: first factors from base A, second from the lane's columns;
// flush(header, sum) takes each output.  Two batches are in flight: while one
// multiplies, the next one's operands and the offsets of the one after load
// (outputs of a stage never read what the stage writes).  About seven
// instructions per FMA, of the 64 issue slots an FP64 instruction takes; with
// packed 10-bit column numbers and absent terms predicated off it was 20, and
// a warp alone reached 12 % of the FP64 pipe.  Queues closed one by one waste
// no FMA on rows of unequal length (four rows in step wasted 10 to 40 %).
template <class Flush>
__device__ __forceinline__ void run_stage(const Stage& st, int warp, const char* A, const char* col,
                                          const Flush& flush) {
  const int nb = st.nb;
  const uint4* pa = st.a + warp * (nb + 1);
  const uint4* pb = st.b + warp * (nb + 1);
  const unsigned* ph = st.h + warp * st.hs;
  double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
  unsigned hd = __ldg(ph);
#define HERM_LOAD(X, wa, wb)                                                                  \
  const uint4 X##w = wb;                                                                      \
  const double X##a0 = lds(A, wa.x), X##b0 = lds(col, wb.x & 0x7FFFFFFFu);                    \
  const double X##a1 = lds(A, wa.y), X##b1 = lds(col, wb.y & 0x7FFFFFFFu);                    \
  const double X##a2 = lds(A, wa.z), X##b2 = lds(col, wb.z & 0x7FFFFFFFu);                    \
  const double X##a3 = lds(A, wa.w), X##b3 = lds(col, wb.w & 0x7FFFFFFFu);
#define HERM_END(w, s)                                                                        \
  if ((int)(w) < 0) {                                                                         \
    flush(hd, s);                                                                             \
    s = 0.0;                                                                                  \
    hd = __ldg(++ph);                                                                         \
  }
#define HERM_FMA(X)                                                                           \
  s0 = fma(X##a0, X##b0, s0);                                                                 \
  s1 = fma(X##a1, X##b1, s1);                                                                 \
  s2 = fma(X##a2, X##b2, s2);                                                                 \
  s3 = fma(X##a3, X##b3, s3);                                                                 \
  if ((int)(X##w.x | X##w.y | X##w.z | X##w.w) < 0) {                                         \
    HERM_END(X##w.x, s0)                                                                      \
    HERM_END(X##w.y, s1)                                                                      \
    HERM_END(X##w.z, s2)                                                                      \
    HERM_END(X##w.w, s3)                                                                      \
  }
  uint4 wa = __ldg(pa), wb = __ldg(pb);
  for (int j = 0; j < nb; j += 2) {
    HERM_LOAD(p, wa, wb)
    const uint4 va = __ldg(pa + j + 1), vb = __ldg(pb + j + 1);
    HERM_LOAD(q, va, vb)
    wa = __ldg(pa + j + 2);
    wb = __ldg(pb + j + 2);
    HERM_FMA(p)
    HERM_FMA(q)
  }
#undef HERM_LOAD
#undef HERM_END
#undef HERM_FMA
}

// store of an output into its column (kScale: times the header's scale
// factor, kAdd: added)
template <bool kScale, bool kAdd>
struct StoreCols {
  char* col;
  const double* pal;
  __device__ __forceinline__ void operator()(unsigned h, double s) const {
    const unsigned d = h & 0xFFFFFu;
    if (kScale && (h >> 20)) s *= __ldg(pal + (h >> 20));
    if (kAdd) s += lds(col, d);
    sts(col, d, s);
  }
};

// y rows staged per warp before their kets are summed
__host__ __device__ constexpr int stage_rows(int nw) { return nw == 1 ? 32 : 16; }

// kMode: bit 0 gamma, bit 1 J, 4 gradient; kNW warps per block.
template <int kMode, int kNW>
__global__ void __launch_bounds__(32 * kNW, 16 / kNW) herm_kernel(const __grid_constant__ HermArgs g) {
  extern __shared__ double sm[];
  constexpr int kRows = stage_rows(kNW);
  constexpr bool kG = (kMode & 1) != 0, kY = (kMode & 6) != 0, kF = (kMode & 4) != 0;
  const int lane = threadIdx.x & 31, warp = kNW > 1 ? threadIdx.x >> 5 : 0;
  const auto sync = [] {
    if (kNW > 1) __syncthreads();
  };
  double* col = sm + lane;
  char* cb = (char*)col;
  const int4 tile = __ldg(g.tiles + blockIdx.x);
  const HermCls& c = g.cls[tile.x];
  const int W = c.W, NP = 32 / W, sub = lane / W;
  const int Lab = c.Lab, lc = c.lc;
  const int q = tile.y + (lane - sub * W);
  const int qc = min(q, c.nket - 1);
  const double Cx = __ldg(c.auxc + 3 * qc), Cy = __ldg(c.auxc + 3 * qc + 1), Cz = __ldg(c.auxc + 3 * qc + 2);
  const int ao = __ldg(c.aux_ao + qc);
  double* PW = col + c.cPW * 32;
  double* XC = col + c.cX * 32;
  double* B = col + c.cB * 32;
  double f0 = 0.0, f1 = 0.0, f2 = 0.0;
  col[c.cZero * 32] = 0.0;
  PW[0] = 1.0;
  PW[(lc + 1) * 32] = 1.0;
  PW[2 * (lc + 1) * 32] = 1.0;
  if (kY) {
    // the ket's q in Cartesian monomials, times their factorials
    for (int n = warp; n < c.ncc; n += kNW) {
      double v = 0.0;
      for (int k = __ldg(c.cptr + n); k < __ldg(c.cptr + n + 1); ++k) {
        const int2 e = __ldg(c.cent + k);
        v = fma(__ldg(c.pal + e.y), __ldg(g.cvec + ao + e.x), v);
      }
      col[(c.cCP + n) * 32] = v;
    }
  }
  if (kG)
    for (int n = warp; n < c.ncc; n += kNW) col[(c.cGA + n) * 32] = 0.0;
  for (int e0 = 0; e0 < tile.w; e0 += NP) {
    const int ie = e0 + sub;
    const int prim = tile.z + min(ie, tile.w - 1);
    const bool act = ie < tile.w && q < __ldg(c.cnt + __ldg(c.primpair + prim));
    const double* pr = c.prim + 4LL * prim;
    const double gam = __ldg(pr);
    const double Rx = __ldg(pr + 1) - Cx, Ry = __ldg(pr + 2) - Cy, Rz = __ldg(pr + 3) - Cz;
    const double R2 = fma(Rz, Rz, fma(Ry, Ry, Rx * Rx));
    if (kNW > 1) __syncthreads(); else __syncwarp();
    if (kG) {
      // the densities of the NP primitive pairs, side by side
      for (int s = 0; s < NP; ++s) {
        const double* H = c.H + (long long)(tile.z + min(e0 + s, tile.w - 1)) * c.nR;
        for (int t = threadIdx.x; t < c.nR; t += 32 * kNW) sm[c.cH * 32 + s * c.nR + t] = __ldg(H + t);
      }
      if (kNW == 1) __syncwarp();
    }
    if (warp == 0) {
      XC[0] = Rx;
      XC[32] = Ry;
      XC[64] = Rz;
    }
    if (warp == 0 && lc > 0) {
      // R_i^j / j!
      double px = Rx, py = Ry, pz = Rz;
      double* P1 = PW + (lc + 1) * 32;
      double* P2 = P1 + (lc + 1) * 32;
      PW[32] = px; P1[32] = py; P2[32] = pz;
      for (int j = 2; j <= lc; ++j) {
        const double ij = c_inv[j];
        px *= Rx * ij; py *= Ry * ij; pz *= Rz * ij;
        PW[j * 32] = px; P1[j * 32] = py; P2[j * 32] = pz;
      }
    }
    for (int ic = 0; ic < c.Kc; ++ic) {
      // geometry, Boys function and R recursion: the first warp (the others
      // wait, and the SM's other blocks run)
      if (ic > 0) sync();
      if (warp == 0) {
        const double zc = __ldg(c.auxrec + ((long long)qc * c.Kc + ic) * kAuxRec);
        const double ccp = __ldg(c.auxrec + ((long long)qc * c.Kc + ic) * kAuxRec + 1);
        const double rs = rsqrt_fp64(gam + zc);
        const double r = rs * rs;
        const double gr = gam * r;
        const double rho = gr * zc;
        const double Tb = rho * R2, n2r = -2.0 * rho;
        double pref = ccp * rs;
        {
          double b = gr;
          for (int e = lc; e; e >>= 1) {
            if (e & 1) pref *= b;
            if (e > 1) b *= b;
          }
        }
        if (!act) pref = 0.0;
        double FL, ex;
        boys_top(g.boys_tab, g.boys_mid, c.boys_cL, c.L, Lab > 0, Tb, FL, ex);
        double fm = pref * FL;
        if (Lab > 0) {
          double b = n2r;
          for (int e = Lab; e; e >>= 1) {
            if (e & 1) fm *= b;
            if (e > 1) b *= b;
          }
          double pe = pref * ex;
          B[0] = pe;
          for (int m = 1; m < Lab; ++m) {
            pe *= n2r;
            B[m * 32] = pe;
          }
        }
        // R_e^(m), |e| <= Lab - m, in place from R^(m+1): degrees descend, so an
        // entry is overwritten only after its last reader.  Operation words:
        // destination, sources, then axis column | factor << 20 | scale << 24
        col[0] = fm;
        for (int m = Lab - 1; m >= 0; --m) {
          const int b1 = c.rbeg[m + 1];
          for (int b = c.rbeg[m]; b < b1; b += 4) {
            double u[4];
            unsigned dst[4];
  #pragma unroll
            for (int k = 0; k < 4; ++k) {
              const uint4 w = __ldg(c.rops + b + k);
              const int kk = (int)((w.w >> 20) & 0xF), id = (int)(w.w >> 24);
              double v = lds(cb, w.z);
              if (kk > 1) v *= c_int[kk];
              u[k] = kk ? fma(lds(cb, w.w & 0xFFFFFu), lds(cb, w.y), v) : lds(cb, w.w & 0xFFFFFu) * lds(cb, w.y);
              if (id) u[k] *= __ldg(c.pal + id);  // 1/e! on the last level
              dst[k] = w.x;
            }
  #pragma unroll
            for (int k = 0; k < 4; ++k) sts(cb, dst[k], u[k]);
          }
          fm = fma(-R2, fm, B[m * 32]) * c_inv[2 * (lc + m) + 1];
          col[0] = fm;
        }
      }
      sync();
      if (kG) {
        run_stage(c.Z, warp, (const char*)(sm + c.cH * 32 + sub * c.nR), cb, StoreCols<true, false>{cb, c.pal});
        sync();
        run_stage(c.gz, warp, cb, cb, StoreCols<false, false>{cb, c.pal});
        sync();
        run_stage(c.gy, warp, cb, cb, StoreCols<false, false>{cb, c.pal});
        sync();
        run_stage(c.gx, warp, cb, cb, StoreCols<false, true>{cb, c.pal});
        sync();
      }
      if (kY) {
        run_stage(c.jx, warp, cb, cb, StoreCols<false, false>{cb, c.pal});
        sync();
        run_stage(c.jy, warp, cb, cb, StoreCols<false, false>{cb, c.pal});
        sync();
        run_stage(c.jw, warp, cb, cb, StoreCols<true, false>{cb, c.pal});
        sync();
        // y_a rows of 32 lanes staged in the B columns (row stride 33); then
        // 32 / rows lanes per row, a power of two, sum the kets of each
        // primitive pair
        double* stg = sm + c.cB * 32 + warp * kRows * 33;
        const double* Hf = kF ? c.H + 3LL * prim * c.nY : nullptr;
        int row = 0, amine = 0;
        const auto drain = [&]() {
          sum_rows(c, stg, row, tile, e0, lane, [&](int r) { return __shfl_sync(0xffffffffu, amine, r); });
          row = 0;
        };
        run_stage(c.Y, warp, cb, cb, [&](unsigned h, double v) {
          stg[row * 33 + lane] = v;
          if (lane == row) amine = (int)(h & 0xFFFF);
          if (kF) {
            const double* hf = Hf + (h & 0xFFFF);
            if (h & 0x10000u) f0 = fma(__ldg(hf), v, f0);
            if (h & 0x20000u) f1 = fma(__ldg(hf + c.nY), v, f1);
            if (h & 0x40000u) f2 = fma(__ldg(hf + 2 * c.nY), v, f2);
          }
          if (++row == kRows) drain();
        });
        if (row) drain();
      }
    }
  }
  if (kG) {
    sync();
    for (int C = warp; C < c.nC && q < c.nket; C += kNW) {
      double v = 0.0;
      for (int k = __ldg(c.gptr + C); k < __ldg(c.gptr + C + 1); ++k) {
        const int2 e = __ldg(c.gent + k);
        v = fma(__ldg(c.pal + e.y), col[(c.cGA + e.x) * 32], v);
      }
      fix_add(g.gacc + kFixWords * (ao + C), v);
    }
  }
  if (kF && q < c.nket) {
    unsigned long long* f = g.facc + kFixWords * 3 * (long long)__ldg(c.aux_atom + qc);
    fix_add(f, -f0);
    fix_add(f + kFixWords, -f1);
    fix_add(f + 2 * kFixWords, -f2);
  }
}

// ---------------------------------------------------------------------------
// per pair: Hermite densities before, J blocks and forces after
// ---------------------------------------------------------------------------

struct HermLabDev {
  double* prim;
  double* scale;
  const int* primab;  // ia Kb + ib of each primitive pair
  double* H;
  unsigned long long* Y;
  int nR, nY;
};

struct HermPairArgs {
  DevBasis orb;
  const int4* pairs;   // {shell a, shell b, Lab, first primitive (within its Lab)}
  const int4* pairs2;  // {AO a, AO b, a == b, its primitive pairs}
  const HermLabDev* lab;
  const double* sph;   // solid-harmonic matrices
  const int* sphoff;
  const double* D;
  long long ldD;
  int chunk;           // primitives of a pair per warp
  unsigned long long* Jacc;
  unsigned long long* facc;
  const int* atom;     // atom of each orbital shell
};

// E~ tables of one primitive pair, E~_t = t! (2 gamma)^t E_t per axis:
//   E~^{i+1,j}_t = t E~_{t-1} + PA E~_t + E~_{t+1} / (2 gamma)
// (j + 1: PB), at E[((axis * (ia + 1) + i) * (ib + 1) + j) * nt + t]; entries
// with t > i + j are zero.  Lanes over (axis, t).
__device__ __forceinline__ void etables(double* E, int ia, int ib, int nt, const double* PA, const double* PB,
                                        double h) {
  const int lane = threadIdx.x;
  const int sj = nt, si = (ib + 1) * nt, sa = (ia + 1) * si;
  for (int i = 0; i <= ia; ++i)
    for (int j = 0; j <= ib; ++j) {
      for (int w = lane; w < 3 * nt; w += 32) {
        const int ax = w / nt, t = w - ax * nt;
        double v = 0.0;
        if (i + j == 0) {
          v = t == 0 ? 1.0 : 0.0;
        } else if (t <= i + j) {
          const double* s = E + ax * sa + (j ? i * si + (j - 1) * sj : (i - 1) * si);
          const double x = j ? PB[ax] : PA[ax];
          v = x * s[t];
          if (t > 0) v = fma((double)t, s[t - 1], v);
          if (t + 1 < nt) v = fma(h, s[t + 1], v);
        }
        E[ax * sa + i * si + j * sj + t] = v;
      }
      __syncwarp();
    }
}

struct PairGeom {
  double za, zb, g, h, K;
  double P[3], PA[3], PB[3];
};

__device__ __forceinline__ PairGeom pair_geom(const DevBasis& o, int sa, int sb, int ia, int ib) {
  PairGeom r;
  const double* A = o.xyz + 3 * sa;
  const double* B = o.xyz + 3 * sb;
  r.za = o.exps[o.off[sa] + ia];
  r.zb = o.exps[o.off[sb] + ib];
  r.g = r.za + r.zb;
  const double ig = 1.0 / r.g;
  r.h = 0.5 * ig;
  double ab2 = 0.0;
  for (int x = 0; x < 3; ++x) {
    const double ab = A[x] - B[x];
    ab2 += ab * ab;
    r.P[x] = (r.za * A[x] + r.zb * B[x]) * ig;
    r.PA[x] = r.P[x] - A[x];
    r.PB[x] = r.P[x] - B[x];
  }
  r.K = o.coefs[o.off[sa] + ia] * o.coefs[o.off[sb] + ib] * exp(-r.za * r.zb * ig * ab2) * 34.98683665524972 * ig;
  return r;
}

// The power of two 2^e by which y_a of degree t is held: about the largest
// |E~^ab_a| it is multiplied by (with 2 gamma, for the forces), so that the
// fixed-point words see the size of its term in J (in the force).  E~_t is the
// mean of the t-th derivative of (x + PA)^i (x + PB)^j over a normal
// distribution of variance h = 1/(2 gamma), i + j = n: about n!/(n - t)! times
// the largest n - t of the factors, each sqrt(|PA|^2 + h (n - t)/e).  (Between
// the tightest and the most diffuse shells it spans h^6.)
__device__ __forceinline__ int potential_scale(int la, int lb, double pa2, double pb2, double h, int t, bool grad) {
  if (grad) ++la;
  const int n = la + lb, m = n - t;
  const float hm = (float)(h * m) * 0.36787944f;
  float ra = (float)pa2 + hm, rb = (float)pb2 + hm;
  const int small = ra < rb ? la : lb;           // factors of the smaller kind
  const int k = max(small - t, 0);               // of them, those left
  float f = 1.0f;
  for (int i = 0; i < t; ++i) f *= (float)(n - i);
  float l = log2f(f) + 0.5f * (k * log2f(fminf(ra, rb)) + (m - k) * log2f(fmaxf(ra, rb)));
  if (m == 0) l = log2f(f);                      // (no factor: the logarithm may be infinite)
  else if (k == 0) l = log2f(f) + 0.5f * m * log2f(fmaxf(ra, rb));
  if (grad) l -= log2f((float)h);
  return (int)rintf(fminf(fmaxf(l, -500.0f), 500.0f));
}

// (y, z) of index w in the graded order of two exponents
__device__ __forceinline__ void yz_of(int w, int& y, int& z) {
  int n = 0;
  while ((n + 1) * (n + 2) / 2 <= w) ++n;
  z = w - n * (n + 1) / 2;
  y = n - z;
}

// The pair's weighted density block in Cartesians: Dc[a][b] = w sum T_Aa D_AB T_Bb
__device__ __forceinline__ void dens_cart(const HermPairArgs& g, int la, int lb, const int4& p2, double* tmp,
                                          double* Dc) {
  const int lane = threadIdx.x;
  const int nA = 2 * la + 1, nB = 2 * lb + 1, na = (la + 1) * (la + 2) / 2, nb = (lb + 1) * (lb + 2) / 2;
  const double* Ta = g.sph + g.sphoff[la];
  const double* Tb = g.sph + g.sphoff[lb];
  const double wt = p2.z ? 1.0 : 2.0;
  for (int w = lane; w < nA * nb; w += 32) {
    const int A = w / nb, b = w - A * nb;
    double v = 0.0;
    for (int B = 0; B < nB; ++B) v = fma(g.D[(long long)(p2.x + A) * g.ldD + p2.y + B], Tb[B * nb + b], v);
    tmp[w] = wt * v;
  }
  __syncwarp();
  for (int w = lane; w < na * nb; w += 32) {
    const int a = w / nb, b = w - a * nb;
    double v = 0.0;
    for (int A = 0; A < nA; ++A) v = fma(Ta[A * na + a], tmp[A * nb + b], v);
    Dc[w] = v;
  }
  __syncwarp();
}

// Cartesian index of (x, y, z)
__device__ __forceinline__ int cidx(int y, int z) {
  const int m = y + z;
  return m * (m + 1) / 2 + z;
}

// M[ty][tz] = sum_{ay, by} Dc[(ax ay az)][(bx by bz)] Ey[ay][by][ty] Ez[az][bz][tz]
__device__ __forceinline__ double dens_yz(const double* Dc, int nb, int da, int db, const double* Ey, const double* Ez,
                                          int si, int sj, int ty, int tz) {
  double v = 0.0;
  for (int ay = 0; ay <= da; ++ay)
    for (int by = 0; by <= db; ++by) {
      const int az = da - ay, bz = db - by;
      if (ay + by < ty || az + bz < tz) continue;
      v = fma(Dc[cidx(ay, az) * nb + cidx(by, bz)] * Ey[ay * si + by * sj + ty], Ez[az * si + bz * sj + tz], v);
    }
  return v;
}

// The per-pair kernels run one warp per shell pair and range of `chunk` of its
// primitives (blockIdx.y).  A warp takes some 10 us a primitive, so pairs of
// many primitives are cut where there are few pairs (one (p p| pair of 256
// primitives: 3.2 ms a build uncut, 0.12 cut); the more ranges, the more
// often the pair's density is transformed and its J block added.
__device__ __forceinline__ int2 prim_range(const HermPairArgs& g, const int4& p2) {
  const int k0 = (int)blockIdx.y * g.chunk;
  return int2{k0, min(p2.w, k0 + g.chunk)};
}

// Primitive records, and with dens the Hermite densities H~_a = K h^|a| sum
// Dc E~_a (gradient: the three arrays of (a_i + 1) H~_a at a + 1_i).
template <bool kGrad>
__global__ void __launch_bounds__(32) herm_pre_kernel(const __grid_constant__ HermPairArgs g, int dens) {
  extern __shared__ double sm[];
  const int lane = threadIdx.x;
  const int4 p1 = __ldg(g.pairs + blockIdx.x), p2 = __ldg(g.pairs2 + blockIdx.x);
  const int la = g.orb.l[p1.x], lb = g.orb.l[p1.y], Kb = g.orb.k[p1.y];
  const HermLabDev L = g.lab[p1.z];
  const int Lab = la + lb, nt = Lab + 1, na = (la + 1) * (la + 2) / 2, nb = (lb + 1) * (lb + 2) / 2, nH = nherm(Lab);
  double* Dc = sm;
  double* E = Dc + na * nb;
  double* Hs = E + 3 * (la + 1) * (lb + 1) * nt;  // also dens_cart's scratch
  const int sj = nt, si = (lb + 1) * nt, sa = (la + 1) * si;
  const int2 kr = prim_range(g, p2);
  if (kr.x >= kr.y) return;
  if (dens) dens_cart(g, la, lb, p2, Hs, Dc);
  for (int k = kr.x; k < kr.y; ++k) {
    const int prim = p1.w + k, ab = __ldg(L.primab + prim);
    const PairGeom pg = pair_geom(g.orb, p1.x, p1.y, ab / Kb, ab % Kb);
    if (lane == 0) {
      double* o = L.prim + 4LL * prim;
      o[0] = pg.g;
      o[1] = pg.P[0]; o[2] = pg.P[1]; o[3] = pg.P[2];
    }
    const int nT = kGrad ? Lab + 2 : Lab + 1;
    if (lane < nT) {
      const double pa2 = pg.PA[0] * pg.PA[0] + pg.PA[1] * pg.PA[1] + pg.PA[2] * pg.PA[2];
      const double pb2 = pg.PB[0] * pg.PB[0] + pg.PB[1] * pg.PB[1] + pg.PB[2] * pg.PB[2];
      const int e = potential_scale(la, lb, pa2, pb2, pg.h, lane, kGrad);
      double s = pg.K, b = pg.h;
      for (int k = lane; k; k >>= 1) {
        if (k & 1) s *= b;
        b *= b;
      }
      double* o = L.scale + 2LL * prim * nT + lane;
      o[0] = ldexp(s, e);
      o[nT] = ldexp(1.0, -e);
    }
    if (!dens) continue;
    __syncwarp();
    etables(E, la, lb, nt, pg.PA, pg.PB, pg.h);
    for (int t = lane; t < nH; t += 32) Hs[t] = 0.0;
    __syncwarp();
    const int nyz = (Lab + 1) * (Lab + 2) / 2;
    for (int w = lane; w < nyz; w += 32) {
      int ty, tz;
      yz_of(w, ty, tz);
      for (int ax = 0; ax <= la; ++ax)
        for (int bx = 0; bx <= lb; ++bx) {
          if (ty + tz > Lab - ax - bx) continue;
          const double M = dens_yz(Dc, nb, la - ax, lb - bx, E + sa, E + 2 * sa, si, sj, ty, tz);
          for (int tx = 0; tx <= ax + bx; ++tx) {
            double* d = Hs + hidx(tx, ty, tz);
            *d = fma(E[ax * si + bx * sj + tx], M, *d);
          }
        }
    }
    __syncwarp();
    if (kGrad) {
      double* o = L.H + 3LL * prim * L.nY;
      for (int t = lane; t < 3 * L.nY; t += 32) o[t] = 0.0;
      __syncwarp();
    }
    for (int w = lane; w < nyz; w += 32) {
      int ty, tz;
      yz_of(w, ty, tz);
      double s = pg.K;
      for (int k = 0; k < ty + tz; ++k) s *= pg.h;
      for (int tx = 0; tx <= Lab - ty - tz; ++tx) {
        const double v = s * Hs[hidx(tx, ty, tz)];
        if (kGrad) {
          double* o = L.H + 3LL * prim * L.nY;
          o[hidx(tx + 1, ty, tz)] = (tx + 1) * v;
          o[L.nY + hidx(tx, ty + 1, tz)] = (ty + 1) * v;
          o[2 * L.nY + hidx(tx, ty, tz + 1)] = (tz + 1) * v;
        } else {
          L.H[(long long)prim * L.nR + hidx(tx, ty, tz)] = v;
        }
        s *= pg.h;
      }
    }
  }
}

// y of one primitive pair, degrees 0..deg, from its fixed-point words.
__device__ __forceinline__ void potentials(const HermLabDev& L, int prim, int deg, double* Ys) {
  const double* inv = L.scale + (2LL * prim + 1) * (deg + 1);
  for (int n = 0; n <= deg; ++n) {
    const double f = __ldg(inv + n);
    for (int t = nherm(n - 1) + threadIdx.x; t < nherm(n); t += 32)
      Ys[t] = f * wide_decode(L.Y + kWideWords * ((long long)prim * L.nY + t));
  }
}

// J block of each pair: J_ab = wj sum over primitives of E~ y, through the
// Cartesian block.
__global__ void __launch_bounds__(32) herm_post_kernel(const __grid_constant__ HermPairArgs g) {
  extern __shared__ double sm[];
  const int lane = threadIdx.x;
  const int4 p1 = __ldg(g.pairs + blockIdx.x), p2 = __ldg(g.pairs2 + blockIdx.x);
  const int la = g.orb.l[p1.x], lb = g.orb.l[p1.y], Kb = g.orb.k[p1.y];
  const HermLabDev L = g.lab[p1.z];
  const int Lab = la + lb, nt = Lab + 1, na = (la + 1) * (la + 2) / 2, nb = (lb + 1) * (lb + 2) / 2;
  double* Jc = sm;
  double* E = Jc + na * nb;
  double* Ys = E + 3 * (la + 1) * (lb + 1) * nt;
  double* Ns = Ys + nherm(Lab);  // [(Lab + 1)(Lab + 2) / 2], also the transform's scratch
  const int sj = nt, si = (lb + 1) * nt, sa = (la + 1) * si;
  const int2 kr = prim_range(g, p2);
  if (kr.x >= kr.y) return;
  for (int w = lane; w < na * nb; w += 32) Jc[w] = 0.0;
  for (int k = kr.x; k < kr.y; ++k) {
    const int prim = p1.w + k, ab = __ldg(L.primab + prim);
    const PairGeom pg = pair_geom(g.orb, p1.x, p1.y, ab / Kb, ab % Kb);
    __syncwarp();
    potentials(L, prim, Lab, Ys);
    etables(E, la, lb, nt, pg.PA, pg.PB, pg.h);
    for (int ax = 0; ax <= la; ++ax)
      for (int bx = 0; bx <= lb; ++bx) {
        const int da = la - ax, db = lb - bx, nyz = (da + db + 1) * (da + db + 2) / 2;
        __syncwarp();
        for (int w = lane; w < nyz; w += 32) {
          int ty, tz;
          yz_of(w, ty, tz);
          double v = 0.0;
          for (int tx = 0; tx <= ax + bx; ++tx) v = fma(E[ax * si + bx * sj + tx], Ys[hidx(tx, ty, tz)], v);
          Ns[w] = v;
        }
        __syncwarp();
        for (int w = lane; w < (da + 1) * (db + 1); w += 32) {
          const int ay = w / (db + 1), by = w - ay * (db + 1), az = da - ay, bz = db - by;
          double v = 0.0;
          for (int ty = 0; ty <= ay + by; ++ty) {
            double u = 0.0;
            for (int tz = 0; tz <= az + bz; ++tz) {
              const int n = ty + tz;
              u = fma(E[2 * sa + az * si + bz * sj + tz], Ns[n * (n + 1) / 2 + tz], u);
            }
            v = fma(E[sa + ay * si + by * sj + ty], u, v);
          }
          Jc[cidx(ay, az) * nb + cidx(by, bz)] += v;
        }
      }
  }
  __syncwarp();
  const int nA = 2 * la + 1, nB = 2 * lb + 1;
  const double* Ta = g.sph + g.sphoff[la];
  const double* Tb = g.sph + g.sphoff[lb];
  const double wj = p2.z ? 0.5 : 1.0;
  double* tmp = E;  // [na][nB]
  for (int w = lane; w < na * nB; w += 32) {
    const int a = w / nB, Bi = w - a * nB;
    double v = 0.0;
    for (int b = 0; b < nb; ++b) v = fma(Jc[a * nb + b], Tb[Bi * nb + b], v);
    tmp[w] = v;
  }
  __syncwarp();
  for (int w = lane; w < nA * nB; w += 32) {
    const int Ai = w / nB, Bi = w - Ai * nB;
    double v = 0.0;
    for (int a = 0; a < na; ++a) v = fma(Ta[Ai * na + a], tmp[a * nB + Bi], v);
    fix_add(g.Jacc + kFixWords * ((long long)(p2.x + Ai) * g.ldD + p2.y + Bi), wj * v);
  }
}

// Forces on the two centres of each pair: with d/dA phi_a = 2 za phi_{a+1} -
// a phi_{a-1} on the E~ tables, dE/dA_i = sum Dc dE~ y; the force along P is
// sum over a of H_a y_{a+1_i}, and dE/dB = dE/dP - dE/dA.
__global__ void __launch_bounds__(32) herm_force_kernel(const __grid_constant__ HermPairArgs g) {
  extern __shared__ double sm[];
  const int lane = threadIdx.x;
  const int4 p1 = __ldg(g.pairs + blockIdx.x), p2 = __ldg(g.pairs2 + blockIdx.x);
  const int la = g.orb.l[p1.x], lb = g.orb.l[p1.y], Kb = g.orb.k[p1.y];
  const HermLabDev L = g.lab[p1.z];
  const int Lab = la + lb, nt = Lab + 2, na = (la + 1) * (la + 2) / 2, nb = (lb + 1) * (lb + 2) / 2;
  double* Dc = sm;
  double* E = Dc + na * nb;                            // (la + 1, lb) tables
  double* F = E + 3 * (la + 2) * (lb + 1) * nt;        // derivative tables, (la, lb)
  double* Ys = F + 3 * (la + 1) * (lb + 1) * nt;       // also dens_cart's scratch
  const int sj = nt, si = (lb + 1) * nt, sa = (la + 2) * si, sf = (la + 1) * si;
  const int2 kr = prim_range(g, p2);
  if (kr.x >= kr.y) return;
  dens_cart(g, la, lb, p2, Ys, Dc);
  double dA[3] = {0.0, 0.0, 0.0}, dP[3] = {0.0, 0.0, 0.0};
  for (int k = kr.x; k < kr.y; ++k) {
    const int prim = p1.w + k, ab = __ldg(L.primab + prim);
    const PairGeom pg = pair_geom(g.orb, p1.x, p1.y, ab / Kb, ab % Kb);
    __syncwarp();
    potentials(L, prim, Lab + 1, Ys);
    etables(E, la + 1, lb, nt, pg.PA, pg.PB, pg.h);
    for (int w = lane; w < 3 * sf; w += 32) {
      const int ax = w / sf, rem = w - ax * sf, i = rem / si, r = rem - i * si;
      double v = 2.0 * pg.za * E[ax * sa + (i + 1) * si + r];
      if (i > 0) v = fma(-(double)i, E[ax * sa + (i - 1) * si + r], v);
      F[w] = v;
    }
    __syncwarp();
    const int nyz = (Lab + 2) * (Lab + 3) / 2;
    for (int w = lane; w < nyz; w += 32) {
      int ty, tz;
      yz_of(w, ty, tz);
      for (int ax = 0; ax <= la; ++ax)
        for (int bx = 0; bx <= lb; ++bx) {
          const int da = la - ax, db = lb - bx;
          if (ty + tz > da + db + 1) continue;
          double N = 0.0, NF = 0.0, NP = 0.0;
          for (int tx = 0; tx <= ax + bx; ++tx) {
            const double e = E[ax * si + bx * sj + tx];
            N = fma(e, Ys[hidx(tx, ty, tz)], N);
            if (ty + tz <= Lab) NP = fma(e * (tx + 1), tx + ty + tz <= Lab ? Ys[hidx(tx + 1, ty, tz)] : 0.0, NP);
          }
          for (int tx = 0; tx <= ax + bx + 1 && tx + ty + tz <= Lab + 1; ++tx)
            NF = fma(F[ax * si + bx * sj + tx], Ys[hidx(tx, ty, tz)], NF);
          double M = 0.0;
          if (ty + tz <= da + db) M = dens_yz(Dc, nb, da, db, E + sa, E + 2 * sa, si, sj, ty, tz);
          dA[0] = fma(M, NF, dA[0]);
          dP[0] = fma(2.0 * pg.g * M, NP, dP[0]);
          // y and z: derivative tables on one axis (one degree higher)
          double My = 0.0, Mz = 0.0, Py = 0.0, Pz = 0.0;
          for (int ay = 0; ay <= da; ++ay)
            for (int by = 0; by <= db; ++by) {
              const int az = da - ay, bz = db - by;
              const double d = Dc[cidx(ay, az) * nb + cidx(by, bz)];
              const int oy = ay * si + by * sj, oz = az * si + bz * sj;
              const double ey = E[sa + oy + ty], ez = E[2 * sa + oz + tz];
              My = fma(d * F[sf + oy + ty], ez, My);
              Mz = fma(d * ey, F[2 * sf + oz + tz], Mz);
              if (ty > 0) Py = fma(d * E[sa + oy + ty - 1] * ty, ez, Py);
              if (tz > 0) Pz = fma(d * ey, E[2 * sa + oz + tz - 1] * tz, Pz);
            }
          dA[1] = fma(My, N, dA[1]);
          dA[2] = fma(Mz, N, dA[2]);
          dP[1] = fma(2.0 * pg.g * Py, N, dP[1]);
          dP[2] = fma(2.0 * pg.g * Pz, N, dP[2]);
        }
    }
  }
#pragma unroll
  for (int x = 0; x < 3; ++x)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      dA[x] += __shfl_xor_sync(0xffffffffu, dA[x], o);
      dP[x] += __shfl_xor_sync(0xffffffffu, dP[x], o);
    }
  if (lane < 3) {
    const double a = lane == 0 ? dA[0] : (lane == 1 ? dA[1] : dA[2]);
    const double p = lane == 0 ? dP[0] : (lane == 1 ? dP[1] : dP[2]);
    fix_add(g.facc + kFixWords * (3LL * __ldg(g.atom + p1.x) + lane), a);
    fix_add(g.facc + kFixWords * (3LL * __ldg(g.atom + p1.y) + lane), p - a);
  }
}

// ---------------------------------------------------------------------------
// host: stage tables of one (Lab, lc)
// ---------------------------------------------------------------------------

struct Row {
  int dst;
  double scale;
  std::vector<std::pair<int, int>> t;
};

struct HostStage {
  std::vector<uint4> a, b;
  std::vector<unsigned> h;
  int nb = 0, hs = 0;
  long long terms = 0, rows = 0, scaled = 0;
};

struct Program {
  int Lab, lc, K, nR, ncc, nC;
  int cX, cPW, cU, cB, cCP, cGA, cZero, ncol, ncol_grad;
  std::vector<uint4> rops;
  std::vector<int> rbeg;
  double rinstr = 0;
  HostStage Z, gz, gy, gx, jx, jy, jw, Y;
  std::vector<int> cptr, gptr, ydeg;
  std::vector<int2> cent, gent;
  std::vector<double> pal;
  double instr_gamma, instr_j, instr_base;  // FP64 instructions per primitive triple
};

struct Pal {
  std::vector<double>& v;
  int id(double x) {
    if (x == 1.0) return 0;
    for (size_t i = 1; i < v.size(); ++i)
      if (v[i] == x) return (int)i;
    v.push_back(x);
    return (int)v.size() - 1;
  }
};

double factorial(int n) {
  double r = 1;
  for (int i = 2; i <= n; ++i) r *= i;
  return r;
}

unsigned col_off(int c) { return (unsigned)(c * kColBytes); }

// kinds of stage: store into columns, (H): first factors indexed in the
// density, (Y): destinations are Hermite indices with their axes
enum StageKind { kCols, kDensity, kRows };

HostStage pack(std::vector<Row> rows, Pal pal, StageKind kind, int zero, const std::vector<std::array<int, 3>>& herm,
               int nw) {
  HostStage s;
  std::stable_sort(rows.begin(), rows.end(), [](const Row& a, const Row& b) { return a.t.size() > b.t.size(); });
  const unsigned z = col_off(zero), za = kind == kDensity ? 0u : z;
  // longest first onto the shortest of the warps' queues, four each
  const int nq = 4 * nw;
  std::vector<std::vector<const Row*>> queue(nq);
  std::vector<size_t> len(nq, 0), at(nq, 0), term(nq, 0);
  for (const Row& r : rows) {
    const int k = (int)(std::min_element(len.begin(), len.end()) - len.begin());
    queue[k].push_back(&r);
    len[k] += r.t.size();
    s.terms += (long long)r.t.size();
    ++s.rows;
    s.scaled += pal.id(r.scale) != 0;
  }
  size_t nb = *std::max_element(len.begin(), len.end());
  nb += nb % 2;
  s.nb = (int)nb;
  std::vector<std::vector<unsigned>> head(nw);
  for (int w = 0; w < nw; ++w) {
    for (size_t j = 0; j < nb; ++j) {
      unsigned x[4] = {za, za, za, za}, y[4] = {z, z, z, z};
      for (int i = 0; i < 4; ++i) {
        const int k = 4 * w + i;
        if (at[k] == queue[k].size()) continue;
        const Row& r = *queue[k][at[k]];
        const auto& t = r.t[term[k]];
        x[i] = kind == kDensity ? (unsigned)(t.first * 8) : col_off(t.first);
        y[i] = col_off(t.second);
        if (++term[k] < r.t.size()) continue;
        y[i] |= kLast;
        ++at[k];
        term[k] = 0;
        if (kind == kRows) {
          unsigned m = 0;
          for (int ax = 0; ax < 3; ++ax)
            if (herm[r.dst][ax] > 0) m |= 1u << ax;
          head[w].push_back((unsigned)r.dst | (m << 16));
        } else {
          head[w].push_back(col_off(r.dst) | ((unsigned)pal.id(r.scale) << 20));
        }
      }
      s.a.push_back(uint4{x[0], x[1], x[2], x[3]});
      s.b.push_back(uint4{y[0], y[1], y[2], y[3]});
    }
    // one batch to fetch past the end
    s.a.push_back(uint4{za, za, za, za});
    s.b.push_back(uint4{z, z, z, z});
    s.hs = std::max(s.hs, (int)head[w].size() + 1);  // and one header
  }
  for (int w = 0; w < nw; ++w) {
    head[w].resize(s.hs, 0u);
    s.h.insert(s.h.end(), head[w].begin(), head[w].end());
  }
  return s;
}

Program build_program(int Lab, int lc, int nw) {
  Program p;
  p.Lab = Lab; p.lc = lc;
  p.K = std::min(Lab, lc);
  const int K = p.K;
  p.nR = nherm(Lab);
  p.ncc = ncart(lc); p.nC = 2 * lc + 1;
  p.pal.assign(1, 1.0);
  Pal pal{p.pal};
  std::vector<std::array<int, 3>> herm(p.nR);
  for (int x = 0; x <= Lab; ++x)
    for (int y = 0; x + y <= Lab; ++y)
      for (int z = 0; x + y + z <= Lab; ++z) herm[hidx(x, y, z)] = {x, y, z};
  auto fac3 = [](int x, int y, int z) { return factorial(x) * factorial(y) * factorial(z); };
  // two-index families of the shift's intermediate columns
  std::map<std::array<int, 3>, int> iU, iZ, iY;  // u; (ux, uy, nz); (ux, ny, nz)
  for (int n = 0; n <= K; ++n)
    for (int i = nherm(n - 1); i < nherm(n); ++i) iU[herm[i]] = i;
  for (int ux = 0; ux <= K; ++ux)
    for (int uy = 0; ux + uy <= K; ++uy)
      for (int nz = 0; ux + uy + nz <= lc; ++nz) { int k = (int)iZ.size(); iZ[{ux, uy, nz}] = k; }
  for (int ux = 0; ux <= K; ++ux)
    for (int ny = 0; ux + ny <= lc; ++ny)
      for (int nz = 0; ux + ny + nz <= lc; ++nz) { int k = (int)iY.size(); iY[{ux, ny, nz}] = k; }
  const int nU = (int)iU.size();
  const int sizeU = std::max(nU, (int)iY.size()), sizeB = std::max({(int)iZ.size(), (nw * stage_rows(nw) * 33 + 31) / 32, Lab + 1});
  int c = p.nR;
  p.cZero = c; c += 1;
  p.cX = c; c += 3;
  p.cPW = c; c += 3 * (lc + 1);
  p.cU = c; c += sizeU;
  p.cB = c; c += sizeB;
  p.cCP = c; c += p.ncc;
  p.ncol_grad = c;
  p.cGA = c; c += p.ncc;
  p.ncol = c;
  auto PW = [&](int axis, int j) { return p.cPW + axis * (lc + 1) + j; };
  // ---- R recursion, level m from level m + 1, degrees descending
  p.rbeg.assign(kMaxDeg + 2, 0);
  std::vector<std::vector<uint4>> lev(std::max(Lab, 1));
  for (int m = 0; m < Lab; ++m)
    for (int n = Lab - m; n >= 1; --n)
      for (int i = nherm(n - 1); i < nherm(n); ++i) {
        const auto& e = herm[i];
        int ax = -1;  // prefer an axis with one quantum (a product), then two (one FMA)
        for (int x = 0; x < 3; ++x)
          if (e[x] > 0 && (ax < 0 || e[x] < e[ax])) ax = x;
        std::array<int, 3> e1 = e, e2 = e;
        e1[ax] -= 1;
        e2[ax] -= 2;
        const int k = e[ax] - 1;
        const unsigned s1 = (unsigned)hidx(e1[0], e1[1], e1[2]), s2 = k > 0 ? (unsigned)hidx(e2[0], e2[1], e2[2]) : 0u;
        const int id = m == 0 ? pal.id(1.0 / fac3(e[0], e[1], e[2])) : 0;
        lev[m].push_back(uint4{col_off(i), col_off((int)s1), col_off((int)s2),
                               col_off(p.cX + ax) | ((unsigned)k << 20) | ((unsigned)id << 24)});
        p.rinstr += 1 + (k > 1) + (id != 0);
      }
  // (level m + 1 follows level m, so that rbeg[m + 1] ends level m)
  for (int m = 0; m < Lab; ++m) {
    p.rbeg[m] = (int)p.rops.size();
    const unsigned z = col_off(p.cZero);
    while (lev[m].size() % 4) lev[m].push_back(uint4{z, z, z, z});
    p.rops.insert(p.rops.end(), lev[m].begin(), lev[m].end());
  }
  for (int m = Lab; m < kMaxDeg + 2; ++m) p.rbeg[m] = (int)p.rops.size();
  // ---- gamma
  std::vector<Row> r;
  for (auto& u : iU) {
    const auto& a = u.first;
    Row w{p.cU + u.second, 1.0 / fac3(a[0], a[1], a[2]), {}};
    const int left = Lab - (a[0] + a[1] + a[2]);
    for (int i = 0; i < nherm(left); ++i) w.t.push_back({hidx(a[0] + herm[i][0], a[1] + herm[i][1], a[2] + herm[i][2]), i});
    r.push_back(w);
  }
  p.Z = pack(r, pal, kDensity, p.cZero, herm, nw);
  r.clear();
  for (auto& z : iZ) {
    const int ux = z.first[0], uy = z.first[1], nz = z.first[2];
    Row w{p.cB + z.second, 1.0, {}};
    for (int uz = 0; uz <= std::min(nz, K - ux - uy); ++uz) w.t.push_back({p.cU + iU.at({ux, uy, uz}), PW(2, nz - uz)});
    r.push_back(w);
  }
  p.gz = pack(r, pal, kCols, p.cZero, herm, nw);
  r.clear();
  for (auto& y : iY) {
    const int ux = y.first[0], ny = y.first[1], nz = y.first[2];
    Row w{p.cU + y.second, 1.0, {}};
    for (int uy = 0; uy <= std::min(ny, K - ux); ++uy) w.t.push_back({p.cB + iZ.at({ux, uy, nz}), PW(1, ny - uy)});
    r.push_back(w);
  }
  p.gy = pack(r, pal, kCols, p.cZero, herm, nw);
  r.clear();
  for (int ny = 0; ny <= lc; ++ny)
    for (int nz = 0; ny + nz <= lc; ++nz) {
      const int nx = lc - ny - nz;
      Row w{p.cGA + cart_index(nx, ny, nz), 1.0, {}};
      for (int ux = 0; ux <= std::min(nx, K); ++ux) w.t.push_back({p.cU + iY.at({ux, ny, nz}), PW(0, nx - ux)});
      r.push_back(w);
    }
  p.gx = pack(r, pal, kCols, p.cZero, herm, nw);
  // ---- J
  r.clear();
  for (auto& y : iY) {
    const int ux = y.first[0], ny = y.first[1], nz = y.first[2], nx = lc - ny - nz;
    r.push_back(Row{p.cU + y.second, 1.0, {{p.cCP + cart_index(nx, ny, nz), PW(0, nx - ux)}}});
  }
  p.jx = pack(r, pal, kCols, p.cZero, herm, nw);
  r.clear();
  for (auto& z : iZ) {
    const int ux = z.first[0], uy = z.first[1], nz = z.first[2];
    Row w{p.cB + z.second, 1.0, {}};
    for (int ny = uy; ux + ny + nz <= lc; ++ny) w.t.push_back({p.cU + iY.at({ux, ny, nz}), PW(1, ny - uy)});
    r.push_back(w);
  }
  p.jy = pack(r, pal, kCols, p.cZero, herm, nw);
  r.clear();
  for (auto& u : iU) {
    const auto& a = u.first;
    Row w{p.cU + u.second, 1.0 / fac3(a[0], a[1], a[2]), {}};
    for (int nz = a[2]; a[0] + a[1] + nz <= lc; ++nz) w.t.push_back({p.cB + iZ.at({a[0], a[1], nz}), PW(2, nz - a[2])});
    r.push_back(w);
  }
  p.jw = pack(r, pal, kCols, p.cZero, herm, nw);
  r.clear();
  for (int i = 0; i < p.nR; ++i) {
    const auto& a = herm[i];
    Row w{i, 1.0, {}};
    for (int ux = 0; ux <= std::min(a[0], K); ++ux)
      for (int uy = 0; uy <= std::min(a[1], K - ux); ++uy)
        for (int uz = 0; uz <= std::min(a[2], K - ux - uy); ++uz)
          w.t.push_back({hidx(a[0] - ux, a[1] - uy, a[2] - uz), p.cU + iU.at({ux, uy, uz})});
    r.push_back(w);
  }
  p.Y = pack(r, pal, kRows, p.cZero, herm, nw);
  for (int i = 0; i < p.nR; ++i) p.ydeg.push_back(herm[i][0] + herm[i][1] + herm[i][2]);
  // ---- ket transforms with the monomials' factorials
  const auto T = solid_matrix(lc);
  p.cptr.push_back(0);
  for (int x = lc; x >= 0; --x)
    for (int y = lc - x; y >= 0; --y) {
      const int n = cart_index(x, y, lc - x - y);
      for (int C = 0; C < p.nC; ++C)
        if (T[C * p.ncc + n] != 0.0) p.cent.push_back(int2{C, pal.id(T[C * p.ncc + n] * fac3(x, y, lc - x - y))});
      p.cptr.push_back((int)p.cent.size());
    }
  p.gptr.push_back(0);
  for (int C = 0; C < p.nC; ++C) {
    for (int x = lc; x >= 0; --x)
      for (int y = lc - x; y >= 0; --y) {
        const int n = cart_index(x, y, lc - x - y);
        if (T[C * p.ncc + n] != 0.0) p.gent.push_back(int2{n, pal.id(T[C * p.ncc + n] * fac3(x, y, lc - x - y))});
      }
    p.gptr.push_back((int)p.gent.size());
  }
  p.instr_base = 32 + 8 + (Lab > 0 ? 8 + 4.0 * Lab : 0) + 6.0 * std::max(0, lc - 1) + p.rinstr;
  p.instr_gamma = (double)(p.Z.terms + p.Z.scaled + p.gz.terms + p.gy.terms + p.gx.terms + p.gx.rows);
  p.instr_j = (double)(p.jx.terms + p.jy.terms + p.jw.terms + p.jw.scaled + p.Y.terms + p.Y.rows * 1.2);
  return p;
}

const Program& program(int Lab, int lc, int nw) {
  static std::mutex mu;
  static std::map<std::tuple<int, int, int>, Program> cache;
  std::lock_guard<std::mutex> lk(mu);
  const auto key = std::make_tuple(Lab, lc, nw);
  auto it = cache.find(key);
  if (it == cache.end()) it = cache.emplace(key, build_program(Lab, lc, nw)).first;
  return it->second;
}

// Byte blob of a program's tables; stage pointers as offsets, relocated on upload.
struct Blob {
  std::vector<char> d;
  template <class T>
  size_t add(const std::vector<T>& v) {
    const size_t off = (d.size() + 15) & ~size_t(15);
    d.resize(off + std::max<size_t>(v.size(), 1) * sizeof(T));
    if (!v.empty()) std::memcpy(d.data() + off, v.data(), v.size() * sizeof(T));
    return off;
  }
};

constexpr int kSmemCta = 232448, kSmemSm = 233472;

}  // namespace

struct HermPlan {
  const lx3c_basis* orb = nullptr;
  const lx3c_basis* aux = nullptr;
  bool grad = false;
  long long nao = 0, npair = 0, nprim = 0;
  struct Tier {
    int smem, nw, Lab;  // nw = 0: the unrolled kernel of this Lab
    long long first, n;
  };
  std::vector<Tier> tiers;
  const PrecomputeJob* jobs = nullptr;  // the ket lists' records
  int njobs = 0;
  long long job_blocks = 0;
  char* arena = nullptr;
  size_t zero_off = 0, zero_bytes = 0;  // the fixed-point y of all primitives
  HermPairArgs pa;
  HermArgs ma;
  int smem_pre = 0, smem_post = 0;
  int nchunk = 1;              // ranges of a pair's primitives (HermPairArgs::chunk)
  double flops = 0, max_adds = 0;
};

void herm_destroy(HermPlan* p) {
  if (!p) return;
  cudaFree(p->arena);
  delete p;
}

int herm_launches(const HermPlan* p) { return 3 + (int)p->tiers.size(); }
double herm_flops(const HermPlan* p) { return p->flops; }
double herm_max_adds(const HermPlan* p) { return p->max_adds; }

double herm_class_flops(int Lab, int lc) {
  if (herm_unrolled(Lab, lc)) {
    const UnrolledCost u = herm_unrolled_cost(Lab, lc);
    return 2.0 * (u.base + u.gamma + u.j);
  }
  const Program& p = program(Lab, lc, 1);
  return 2.0 * (p.instr_base + p.instr_gamma + p.instr_j);
}

int herm_build(HermPlan** out, const lx3c_basis* orb, const lx3c_basis* aux, const std::vector<HermBra>& bras,
               const std::vector<HermKet>& kets, bool (*use)(const HermBra&, const HermKet&), HermKeep keep, double tol,
               bool grad, long long nao, cudaStream_t st) {
  *out = nullptr;
  DevState* ds;
  int rc = device_state_get(&ds);
  if (rc) return rc;
  std::unique_ptr<HermPlan, void (*)(HermPlan*)> p(new HermPlan, herm_destroy);
  p->orb = orb; p->aux = aux; p->grad = grad; p->nao = nao;
  // pairs by Lab, most strongly coupled first, so that the pairs keeping a
  // given ket are a prefix
  struct PairRef { double q; int bra, i; };
  std::map<int, std::vector<PairRef>> byL;
  for (size_t b = 0; b < bras.size(); ++b) {
    bool any = false;
    for (auto& k : kets) any = any || use(bras[b], k);
    if (!any) continue;
    for (size_t i = 0; i < bras[b].q.size(); ++i)
      for (auto& k : kets)
        if (use(bras[b], k) && keep(bras[b].q[i], k.q, tol) > 0) {
          byL[bras[b].la + bras[b].lb].push_back(PairRef{bras[b].q[i], (int)b, (int)i});
          break;
        }
  }
  if (byL.empty() || kets.empty()) return LX3C_OK;
  std::vector<int> ao(orb->nshell + 1, 0), aq(aux->nshell + 1, 0);
  for (int64_t s = 0; s < orb->nshell; ++s) ao[s + 1] = ao[s] + 2 * orb->l[s] + 1;
  for (int64_t s = 0; s < aux->nshell; ++s) aq[s + 1] = aq[s] + 2 * aux->l[s] + 1;
  Blob blob;
  std::vector<int4> pairs, pairs2;
  struct LabHost {
    int Lab;
    long long nprim = 0;
    std::vector<PairRef> pr;
    std::vector<long long> prim0;  // first primitive of each pair, and the end
    std::vector<int> primab, primpair;
    size_t H, Y, prim, scale, o_ab, o_pair;  // arena offsets
  };
  std::vector<LabHost> labs;
  std::vector<int> laboff(kMaxDeg + 2, -1);
  int smem_pre = 0, smem_post = 0;
  for (auto& kv : byL) {
    LabHost L;
    L.Lab = kv.first;
    L.pr = std::move(kv.second);
    std::stable_sort(L.pr.begin(), L.pr.end(), [](const PairRef& a, const PairRef& b) { return a.q > b.q; });
    laboff[L.Lab] = (int)labs.size();
    for (size_t i = 0; i < L.pr.size(); ++i) {
      const HermBra& b = bras[L.pr[i].bra];
      const int sa = b.pairs[2 * L.pr[i].i], sb = b.pairs[2 * L.pr[i].i + 1];
      if (L.nprim > 0x7fffffffLL) {
        set_last_error("dfj: too many primitive pairs");
        return LX3C_ENOTSUP;
      }
      L.prim0.push_back(L.nprim);
      pairs.push_back(int4{sa, sb, laboff[L.Lab], (int)L.nprim});
      {
        // the contributing primitive pairs
        double ab2 = 0, q[LX3C_KMAX * LX3C_KMAX], K[LX3C_KMAX * LX3C_KMAX], qmax = 0;
        for (int x = 0; x < 3; ++x) {
          const double d = orb->xyz[3 * sa + x] - orb->xyz[3 * sb + x];
          ab2 += d * d;
        }
        for (int ia = 0; ia < b.Ka; ++ia)
          for (int ib = 0; ib < b.Kb; ++ib) {
            const int r = ia * b.Kb + ib;
            q[r] = prim_bound(orb->exps[orb->off[sa] + ia], orb->coefs[orb->off[sa] + ia], orb->exps[orb->off[sb] + ib],
                              orb->coefs[orb->off[sb] + ib], ab2, b.la, b.lb, &K[r]);
            qmax = std::max(qmax, q[r]);
          }
        for (int r = 0; r < b.Ka * b.Kb; ++r)
          if (prim_kept(K[r], q[r], qmax)) {
            L.primab.push_back(r);
            L.primpair.push_back((int)i);
          }
      }
      pairs2.push_back(int4{ao[sa], ao[sb], sa == sb ? 1 : 0, (int)((long long)L.primab.size() - L.nprim)});
      L.nprim = (long long)L.primab.size();
      const int la = b.la, lb = b.lb, na = ncart(la), nb = ncart(lb), nt = L.Lab + 1;
      const int scr = std::max(nherm(L.Lab), (2 * la + 1) * nb);
      if (grad) {
        const int nt2 = nt + 1;
        smem_pre = std::max(smem_pre, na * nb + 3 * (la + 1) * (lb + 1) * nt + scr);
        smem_post = std::max(smem_post, na * nb + 3 * (2 * la + 3) * (lb + 1) * nt2 +
                                            std::max(nherm(L.Lab + 1), (2 * la + 1) * nb));
      } else {
        smem_pre = std::max(smem_pre, na * nb + 3 * (la + 1) * (lb + 1) * nt + scr);
        smem_post = std::max(smem_post, na * nb + std::max(3 * (la + 1) * (lb + 1) * nt + nherm(L.Lab) +
                                                               (L.Lab + 1) * (L.Lab + 2) / 2,
                                                           na * (2 * lb + 1)));
      }
    }
    L.prim0.push_back(L.nprim);
    p->nprim += L.nprim;
    labs.push_back(std::move(L));
  }
  p->npair = (long long)pairs.size();
  // ranges of primitives: 16 warps an SM's worth of them, four or more each
  const int per = (int)std::max<long long>(4, p->nprim / (dev_nsm(ds) * 16));
  int most = 1;
  for (const int4& q : pairs2) most = std::max(most, q.w);
  p->nchunk = (most + per - 1) / per;
  p->pa.chunk = per;
  p->smem_pre = smem_pre * 8;
  p->smem_post = smem_post * 8;
  // classes and their tables
  struct ClsHost {
    HermCls c;
    int lab, ket;
    size_t rops, cptr, cent, gptr, gent, pal, ydeg, cnt, st[8][3];
    std::vector<int> counts;
    double instr;
    int smem;
  };
  std::vector<ClsHost> cls;
  std::map<std::pair<int, int>, int> first_of;  // tables shared by classes of one program
  double total = 0;
  for (size_t li = 0; li < labs.size(); ++li)
    for (size_t ki = 0; ki < kets.size(); ++ki) {
      const LabHost& L = labs[li];
      const HermKet& k = kets[ki];
      ClsHost x;
      x.lab = (int)li; x.ket = (int)ki;
      x.counts.resize(L.pr.size());
      double tri = 0;
      std::vector<char> used(bras.size());
      for (size_t b = 0; b < bras.size(); ++b) used[b] = use(bras[b], k);
      for (size_t i = 0; i < L.pr.size(); ++i) {
        x.counts[i] = used[L.pr[i].bra] ? keep(L.pr[i].q, k.q, tol) : 0;
        tri += (double)x.counts[i] * (double)(L.prim0[i + 1] - L.prim0[i]);
      }
      if (tri == 0) continue;
      const int Lp = L.Lab + (grad ? 1 : 0);
      // warps per block: as many as it takes to reach eight on an SM (asking
      // for 12 or 16 leaves short stages with idle queues: DF-J of 32 atoms
      // 105 -> 109 and 122 ms; one warp throughout: 110 ms)
      const Program& p1 = program(Lp, k.lc, 1);
      const int fit = kSmemSm / ((grad ? p1.ncol_grad : p1.ncol) * kColBytes + 2048);
      const bool unr = herm_unrolled(Lp, k.lc);
      const int nw = unr ? 0 : (fit >= 8 ? 1 : (fit >= 4 ? 2 : 4));  // 0: the unrolled kernel
      const Program& pg = program(Lp, k.lc, std::max(nw, 1));
      HermCls& c = x.c;
      std::memset(&c, 0, sizeof(c));
      c.nw = nw;
      c.Lab = Lp; c.lc = k.lc; c.Kc = k.Kc; c.L = Lp + k.lc; c.nR = pg.nR; c.nY = pg.nR; c.ncc = pg.ncc; c.nC = pg.nC;
      c.nket = (int)k.shells.size();
      c.cX = pg.cX; c.cPW = pg.cPW; c.cU = pg.cU; c.cB = pg.cB; c.cCP = pg.cCP; c.cGA = pg.cGA;
      c.cZero = pg.cZero;
      c.cH = grad ? pg.ncol_grad : pg.ncol;
      for (int m = 0; m < kMaxDeg + 2; ++m) c.rbeg[m] = pg.rbeg[m];
      c.boys_cL = boys_large_const(c.L);
      const UnrolledCost uc = unr ? herm_unrolled_cost(Lp, k.lc)
                                  : UnrolledCost{pg.instr_base, pg.instr_gamma, pg.instr_j};
      x.instr = (uc.base + uc.j + (grad ? 3.0 * pg.nR : uc.gamma)) * k.Kc;
      // W kets side by side: the widest power of two whose ragged end wastes
      // least (narrower tiles pay one more y row sum per primitive pair), of
      // those whose 32 / W densities fit beside the columns (one ket at a time
      // takes 116 KB of them at degree 12)
      const auto smem_of = [&](int W) {
        return unr ? herm_unrolled_smem(Lp, k.lc, W) : c.cH * kColBytes + (grad ? 0 : 32 / W * pg.nR * 8);
      };
      double best = 1e300;
      for (int W = 32; W >= 1 && smem_of(W) <= kSmemCta; W /= 2) {
        double slots = 0;
        for (size_t i = 0; i < L.pr.size(); ++i)
          slots += (double)((x.counts[i] + W - 1) / W * W) * (double)(L.prim0[i + 1] - L.prim0[i]);
        const double cost = slots * (1.0 + 0.02 * (32 / W - 1));
        if (cost < best * 0.999) { best = cost; c.W = W; }
      }
      if (!c.W) {
        set_last_error("dfj: Hermite class does not fit in shared memory");
        return LX3C_ENOTSUP;
      }
      x.smem = smem_of(c.W);
      p->flops += 2.0 * x.instr * tri;
      total += x.instr * best / 32.0;
      auto key = std::make_pair(Lp, k.lc);  // (nw follows from them)
      if (first_of.count(key)) {
        const ClsHost& f = cls[first_of[key]];
        x.rops = f.rops; x.cptr = f.cptr; x.cent = f.cent; x.gptr = f.gptr; x.gent = f.gent; x.pal = f.pal; x.ydeg = f.ydeg;
        std::memcpy(x.st, f.st, sizeof(x.st));
      } else {
        first_of[key] = (int)cls.size();
        x.rops = unr ? 0 : blob.add(pg.rops); x.cptr = blob.add(pg.cptr); x.cent = blob.add(pg.cent); x.gptr = blob.add(pg.gptr);
        x.gent = blob.add(pg.gent); x.pal = blob.add(pg.pal); x.ydeg = blob.add(pg.ydeg);
        const HostStage* hs[8] = {&pg.Z, &pg.gz, &pg.gy, &pg.gx, &pg.jx, &pg.jy, &pg.jw, &pg.Y};
        std::memset(x.st, 0, sizeof(x.st));
        for (int s = 0; s < 8 && !unr; ++s) {
          x.st[s][0] = blob.add(hs[s]->a);
          x.st[s][1] = blob.add(hs[s]->b);
          x.st[s][2] = blob.add(hs[s]->h);
        }
      }
      {
        const HostStage* hs[8] = {&pg.Z, &pg.gz, &pg.gy, &pg.gx, &pg.jx, &pg.jy, &pg.jw, &pg.Y};
        Stage* ds_[8] = {&c.Z, &c.gz, &c.gy, &c.gx, &c.jx, &c.jy, &c.jw, &c.Y};
        for (int s = 0; s < 8; ++s) {
          ds_[s]->nb = hs[s]->nb;
          ds_[s]->hs = hs[s]->hs;
        }
      }
      x.cnt = blob.add(x.counts);
      cls.push_back(std::move(x));
    }
  if (cls.empty()) return LX3C_OK;
  // tiles: about eight per resident warp slot overall, at least one block of
  // kets wide; a tile runs up to 64 groups of primitive pairs so that the
  // kets' gamma is flushed rarely
  std::vector<int> order(cls.size());
  for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
  auto occ = [&](int smem) { return std::min(32, kSmemSm / (smem + 1024)); };
  // classes of equal block size and occupancy share a launch, the largest
  // footprint first
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
    if (cls[a].c.nw != cls[b].c.nw) return cls[a].c.nw > cls[b].c.nw;
    if (!cls[a].c.nw)
      return cls[a].c.Lab != cls[b].c.Lab ? cls[a].c.Lab > cls[b].c.Lab : cls[a].instr > cls[b].instr;
    const int oa = occ(cls[a].smem), ob = occ(cls[b].smem);
    return oa != ob ? oa < ob : cls[a].instr > cls[b].instr;
  });
  std::vector<int4> tiles;
  int natom = 1;
  for (int a : orb->atom) natom = std::max(natom, a + 1);
  for (int a : aux->atom) natom = std::max(natom, a + 1);
  std::vector<double> adds(natom, 0.0);  // contributions to each atom's force accumulators
  const double target = total / (dev_nsm(ds) * 8 * 16.0);
  int bin = -1;
  const int bins[] = {1, 2, 3, 4, 6, 8, 12, 16, 24, 32};
  for (int ci : order) {
    ClsHost& x = cls[ci];
    const LabHost& L = labs[x.lab];
    int b = 0;
    while (x.c.nw && b + 1 < 10 && bins[b + 1] <= occ(x.smem)) ++b;
    if (!x.c.nw) b = 100 + x.c.Lab;  // one launch per Lab
    if (b != bin || p->tiers.back().nw != x.c.nw) {
      p->tiers.push_back(HermPlan::Tier{0, x.c.nw, x.c.Lab, (long long)tiles.size(), 0});
      bin = b;
    }
    HermPlan::Tier& t = p->tiers.back();
    t.smem = std::max(t.smem, x.smem);
    const int W = x.c.W, NP = 32 / W;
    // a tile ends with three atomics for each of a lane's sums (a ket's gamma, or
    // its force), which cost the chip about as much as 30 FP64 instructions
    // each: tiles of one or two primitives on light classes are mostly flushes
    // (20 contracted p shells over 160 kets, gamma alone 1.18 ms), so a tile has
    // work for as much, if that leaves a warp for each slot (0.76; for three
    // times as much 0.44, but DF-J of 4 atoms 1.70 -> 1.78)
    const double flush = 30.0 * 3.0 * (grad ? 3 : x.c.nC);
    const double work = std::max(target, std::min(flush, 16.0 * target));
    const long long step = NP * std::max<long long>(1, std::min<long long>(64, (long long)(work / x.instr + 0.5)));
    for (int k0 = 0; k0 < x.c.nket; k0 += W) {
      // pairs keeping ket k0: a prefix, save for pairs this class does not use
      size_t np = x.counts.size();
      while (np > 0 && x.counts[np - 1] <= k0) --np;
      const long long ne = L.prim0[np];
      for (long long e = 0; e < ne; e += step)
        tiles.push_back(int4{ci, k0, (int)e, (int)std::min<long long>(step, ne - e)});
      if (grad)  // one contribution per axis from each lane with the ket, of each warp
        for (int q = k0; q < std::min(k0 + W, x.c.nket); ++q)
          adds[aux->atom[kets[x.ket].shells[q]]] += (double)((ne + step - 1) / step) * NP * std::max(x.c.nw, 1);
    }
    t.n = (long long)tiles.size() - t.first;
  }
  for (auto& t : p->tiers)
    if (t.n > 0x7fffffffLL) {
      set_last_error("dfj: too many tiles");
      return LX3C_ENOTSUP;
    }
  if (grad) {
    for (const int4& q : pairs)
      for (int s : {q.x, q.y}) adds[orb->atom[s]] += p->nchunk;
    p->max_adds = *std::max_element(adds.begin(), adds.end());
  }
  // ---- one allocation: tables and lists (uploaded), then the work buffers
  std::vector<double> sph;
  std::vector<int> sphoff;
  int lmax = 0;
  for (auto& b : bras) lmax = std::max({lmax, b.la, b.lb});
  for (int l = 0; l <= lmax; ++l) {
    sphoff.push_back((int)sph.size());
    const auto T = solid_matrix(l);
    sph.insert(sph.end(), T.begin(), T.end());
  }
  for (auto& L : labs) {
    L.o_ab = blob.add(L.primab);
    L.o_pair = blob.add(L.primpair);
  }
  const size_t o_sph = blob.add(sph), o_sphoff = blob.add(sphoff);
  const size_t o_pairs = blob.add(pairs), o_pairs2 = blob.add(pairs2), o_tiles = blob.add(tiles);
  const size_t o_atom = blob.add(orb->atom);
  struct KetOff { size_t shells, ao, atom, rec, xyz; };
  std::vector<KetOff> ko(kets.size());
  for (size_t k = 0; k < kets.size(); ++k) {
    std::vector<int> a, t;
    for (int s : kets[k].shells) {
      a.push_back(aq[s]);
      t.push_back(aux->atom[s]);
    }
    ko[k].shells = blob.add(kets[k].shells);
    ko[k].ao = blob.add(a);
    ko[k].atom = blob.add(t);
  }
  std::vector<HermLabDev> ld(labs.size());
  const size_t o_lab = blob.add(ld);
  std::vector<HermCls> hc(cls.size());
  const size_t o_cls = blob.add(hc);
  std::vector<PrecomputeJob> jobs(kets.size());
  const size_t o_jobs = blob.add(jobs);
  size_t top = blob.d.size();
  auto take = [&](size_t bytes) {
    top = (top + 255) & ~size_t(255);
    const size_t o = top;
    top += bytes;
    return o;
  };
  for (size_t k = 0; k < kets.size(); ++k) {
    ko[k].rec = take(kets[k].shells.size() * kets[k].Kc * kAuxRec * 8);
    ko[k].xyz = take(kets[k].shells.size() * 24);
  }
  for (auto& L : labs) {
    const long long nY = nherm(L.Lab + (grad ? 1 : 0));
    L.prim = take((size_t)L.nprim * 32);
    L.scale = take((size_t)L.nprim * 2 * (L.Lab + (grad ? 2 : 1)) * 8);
    L.H = take((size_t)L.nprim * (grad ? 3 * nY : nY) * 8);
  }
  p->zero_off = take(0);
  for (auto& L : labs) L.Y = take((size_t)L.nprim * nherm(L.Lab + (grad ? 1 : 0)) * kWideBytes);
  p->zero_bytes = top - p->zero_off;
  if (cudaMalloc(&p->arena, top) != cudaSuccess) {
    cudaGetLastError();
    set_last_error("dfj: Hermite work buffers do not fit in device memory");
    return LX3C_ENOMEM;
  }
  char* A = p->arena;
  for (size_t i = 0; i < labs.size(); ++i) {
    const LabHost& L = labs[i];
    ld[i].prim = (double*)(A + L.prim);
    ld[i].scale = (double*)(A + L.scale);
    ld[i].primab = (const int*)(A + L.o_ab);
    ld[i].H = (double*)(A + L.H);
    ld[i].Y = (unsigned long long*)(A + L.Y);
    ld[i].nR = nherm(L.Lab);
    ld[i].nY = nherm(L.Lab + (grad ? 1 : 0));
  }
  std::memcpy(blob.d.data() + o_lab, ld.data(), ld.size() * sizeof(HermLabDev));
  for (size_t i = 0; i < cls.size(); ++i) {
    HermCls& c = cls[i].c;
    const ClsHost& x = cls[i];
    Stage* s[8] = {&c.Z, &c.gz, &c.gy, &c.gx, &c.jx, &c.jy, &c.jw, &c.Y};
    for (int k = 0; k < 8; ++k) {
      s[k]->a = (const uint4*)(A + x.st[k][0]);
      s[k]->b = (const uint4*)(A + x.st[k][1]);
      s[k]->h = (const unsigned*)(A + x.st[k][2]);
    }
    c.rops = (const uint4*)(A + x.rops);
    c.cptr = (const int*)(A + x.cptr); c.cent = (const int2*)(A + x.cent);
    c.gptr = (const int*)(A + x.gptr); c.gent = (const int2*)(A + x.gent);
    c.pal = (const double*)(A + x.pal);
    c.ydeg = (const int*)(A + x.ydeg);
    c.cnt = (const int*)(A + x.cnt);
    const LabHost& L = labs[x.lab];
    c.prim = (const double*)(A + L.prim);
    c.scale = (const double*)(A + L.scale);
    c.primpair = (const int*)(A + L.o_pair);
    c.H = (const double*)(A + L.H);
    c.Yacc = (unsigned long long*)(A + L.Y);
    c.auxrec = (const double*)(A + ko[x.ket].rec);
    c.auxc = (const double*)(A + ko[x.ket].xyz);
    c.aux_ao = (const int*)(A + ko[x.ket].ao);
    c.aux_atom = (const int*)(A + ko[x.ket].atom);
    hc[i] = c;
  }
  std::memcpy(blob.d.data() + o_cls, hc.data(), hc.size() * sizeof(HermCls));
  for (size_t k = 0; k < kets.size(); ++k) {
    jobs[k] = PrecomputeJob{nullptr, 0, 1, 1, nullptr, nullptr, (const int32_t*)(A + ko[k].shells),
                            (long long)kets[k].shells.size(), kets[k].Kc, (double*)(A + ko[k].rec),
                            (double*)(A + ko[k].xyz), p->job_blocks};
    p->job_blocks += jobs[k].blocks();
  }
  std::memcpy(blob.d.data() + o_jobs, jobs.data(), jobs.size() * sizeof(PrecomputeJob));
  p->jobs = (const PrecomputeJob*)(A + o_jobs);
  p->njobs = (int)jobs.size();
  HermPairArgs& pa = p->pa;
  pa.orb = orb->dev();
  pa.pairs = (const int4*)(A + o_pairs);
  pa.pairs2 = (const int4*)(A + o_pairs2);
  pa.lab = (const HermLabDev*)(A + o_lab);
  pa.sph = (const double*)(A + o_sph);
  pa.sphoff = (const int*)(A + o_sphoff);
  pa.ldD = nao;
  pa.atom = (const int*)(A + o_atom);
  HermArgs& ma = p->ma;
  ma.cls = (const HermCls*)(A + o_cls);
  ma.tiles = (const int4*)(A + o_tiles);
  ma.boys_tab = dev_boys_tab(ds);
  ma.boys_mid = dev_boys_mid(ds);
  cudaError_t e = cudaMemcpyAsync(A, blob.d.data(), blob.d.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = herm_unrolled_setup();
  const void* kernels[] = {(const void*)herm_kernel<1, 1>, (const void*)herm_kernel<1, 2>, (const void*)herm_kernel<1, 4>,
                           (const void*)herm_kernel<2, 1>, (const void*)herm_kernel<2, 2>, (const void*)herm_kernel<2, 4>,
                           (const void*)herm_kernel<3, 1>, (const void*)herm_kernel<3, 2>, (const void*)herm_kernel<3, 4>,
                           (const void*)herm_kernel<4, 1>, (const void*)herm_kernel<4, 2>, (const void*)herm_kernel<4, 4>};
  for (const void* f : kernels)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCta);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(herm_pre_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCta);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(herm_pre_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCta);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(herm_post_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCta);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(herm_force_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCta);
  if (e != cudaSuccess) {
    set_last_error(std::string("dfj: Hermite plan: ") + cudaGetErrorString(e));
    return LX3C_ECUDA;
  }
  *out = p.release();
  return LX3C_OK;
}

namespace {

dim3 pair_grid(const HermPlan* p) { return dim3((unsigned)p->npair, (unsigned)p->nchunk); }

cudaError_t herm_begin(HermPlan* p, const double* D, bool dens, bool y, cudaStream_t st) {
  cudaError_t e = cudaSuccess;
  if (y) e = cudaMemsetAsync(p->arena + p->zero_off, 0, p->zero_bytes, st);
  if (e == cudaSuccess) e = launch_precompute_jobs(p->orb->dev(), p->aux->dev(), p->jobs, p->njobs, p->job_blocks, st);
  if (e != cudaSuccess) return e;
  HermPairArgs a = p->pa;
  a.D = D;
  if (p->grad)
    herm_pre_kernel<true><<<pair_grid(p), 32, p->smem_pre, st>>>(a, dens ? 1 : 0);
  else
    herm_pre_kernel<false><<<pair_grid(p), 32, p->smem_pre, st>>>(a, dens ? 1 : 0);
  return cudaGetLastError();
}

template <int kMode>
cudaError_t herm_tiles(HermPlan* p, HermArgs a, cudaStream_t st) {
  for (auto& t : p->tiers) {
    a.tiles = p->ma.tiles + t.first;
    if (t.nw == 0) {
      const cudaError_t e = launch_herm_unrolled(t.Lab, a, kMode, t.smem, t.n, st);
      if (e != cudaSuccess) return e;
    } else if (t.nw == 1) herm_kernel<kMode, 1><<<(unsigned)t.n, 32, t.smem, st>>>(a);
    else if (t.nw == 2) herm_kernel<kMode, 2><<<(unsigned)t.n, 64, t.smem, st>>>(a);
    else herm_kernel<kMode, 4><<<(unsigned)t.n, 128, t.smem, st>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t herm_execute(HermPlan* p, const double* D, const double* c, unsigned long long* gacc,
                         unsigned long long* Jacc, cudaStream_t st) {
  cudaError_t e = herm_begin(p, D, gacc != nullptr, Jacc != nullptr, st);
  if (e != cudaSuccess) return e;
  HermArgs a = p->ma;
  a.cvec = c;
  a.gacc = gacc;
  a.facc = nullptr;
  if (gacc && Jacc) e = herm_tiles<3>(p, a, st);
  else if (gacc) e = herm_tiles<1>(p, a, st);
  else e = herm_tiles<2>(p, a, st);
  if (e != cudaSuccess || !Jacc) return e;
  HermPairArgs b = p->pa;
  b.Jacc = Jacc;
  herm_post_kernel<<<pair_grid(p), 32, p->smem_post, st>>>(b);
  return cudaGetLastError();
}

cudaError_t herm_gradient(HermPlan* p, const double* D, const double* c, unsigned long long* facc, cudaStream_t st) {
  cudaError_t e = herm_begin(p, D, true, true, st);
  if (e != cudaSuccess) return e;
  HermArgs a = p->ma;
  a.cvec = c;
  a.gacc = nullptr;
  a.facc = facc;
  e = herm_tiles<4>(p, a, st);
  if (e != cudaSuccess) return e;
  HermPairArgs b = p->pa;
  b.D = D;
  b.facc = facc;
  herm_force_kernel<<<pair_grid(p), 32, p->smem_post, st>>>(b);
  return cudaGetLastError();
}

}  // namespace lx3c
