// Device kernels for contracted 3-center Coulomb integrals (ab|C)
// (arXiv:2210.03192, HGPA scheme of Sec. 2.5.1):
//   precompute_kernel  primitive-pair records gamma, P, PA, K_ab (Appendix A) and
//                    ket primitive records; precompute_jobs_kernel many lists
//   eri3c_kernel     per tile of (one pair, T ket shells):
//                      [00|0]^(m) from the Boys function       Sec. 2.5.2
//                      VRR1                                      Eq. vrr1
//                      CVRR2 prerequisites, contracted early     Eq. a0cv2 / Sec. 2.5.4
//                      CVRR2 targets (n-quantum form) on a solid-
//                      harmonic ket                              Sec. 2.5.4, 2.5.1
//                      HRR                                       Eq. hrr
//                      optional solid-harmonic bra, store
//
// GB300 design notes.  FP64 is the only scarce resource on this part (about
// 2 DFMA per clock per SM against 128 FFMA), so every stage is written to
// issue only the FP64 operations of the FLOP-minimal scheme with all 32 lanes
// busy, while index decoding, shared-memory traffic and table reads (integer,
// load/store pipes) hide under the FP64 pipe.  Each stage is a flat loop over
// (triple block, target) items driven by host-built tables; the triple index
// is the fastest lane index when a tile holds >= 32 triples (warp-uniform table
// entries, conflict-free strided shared memory) and the target index otherwise.
// An item is one target of up to four triples: one decoded table entry and one
// set of addresses serve them all (one triple per item took 47 instructions per
// FP64 instruction at (ff|g), three quarters of the issue slots).
// Primitive contraction happens in shared-memory accumulators (the CVRR2
// prerequisites), so no intermediate CVRR2 value is ever stored to global
// memory and no atomics are needed.
#include <cuda_runtime.h>

#include "boys_device.cuh"
#include "fixed128.cuh"
#include "harmonic_weights.h"
#include "lx3c_internal.h"

namespace lx3c {

__constant__ double c_inv2m1[32];  // 1/(2m+1)

__constant__ double c_q[36] = LX3C_QTABLE;

template <int N>
struct Int {
  static constexpr int n = N;
};

struct FDiv {
  unsigned d, m;
  __device__ __forceinline__ void init(unsigned dd) {
    d = dd;
    m = (dd <= 1u) ? 0u : (0xFFFFFFFFu / dd + 1u);
  }
  // exact for n * d < 2^32
  __device__ __forceinline__ unsigned div(unsigned n) const { return d <= 1u ? n : __umulhi(n, m); }
};

// Compensated dot product (Ogita, Rump and Oishi's Dot2: TwoProduct by FMA,
// TwoSum, errors summed separately): about twice the working precision for
// the same result, at ~10 FP64 operations per term instead of one FMA.
// Explicitly rounded intrinsics keep the compiler from contracting the
// error-free transformations.
struct Dot2 {
  double s, c;
  __device__ __forceinline__ Dot2() : s(0.0), c(0.0) {}
  __device__ __forceinline__ void add(double a, double b) {
    const double p = __dmul_rn(a, b);
    const double ep = fma(a, b, -p);
    const double t = __dadd_rn(s, p);
    const double z = __dsub_rn(t, s);
    const double es = __dadd_rn(__dsub_rn(s, __dsub_rn(t, z)), __dsub_rn(p, z));
    s = t;
    c = __dadd_rn(c, __dadd_rn(ep, es));
  }
  __device__ __forceinline__ double value() const { return __dadd_rn(s, c); }
};

// One FP64 tensor-core step D = A B + C on an 8x8x4 tile, one warp
// (mma.sync m8n8k4 .f64).  With g = lane / 4 and q = lane % 4 the lane holds
// A[g][q], B[q][g] and the accumulator elements C[g][2q], C[g][2q+1].
__device__ __forceinline__ void dmma_8x8x4(double a, double b, double& c0, double& c1) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};\n"
               : "+d"(c0), "+d"(c1)
               : "d"(a), "d"(b));
}

// pref * F_m(T) for m = hi down to lo, written to v[(m - lo) * stride].
// F_hi and exp(-T) come from the interpolation table (T < 2^24; exp(-T) = 0
// from 117 on) or the asymptotic form beyond; lower orders by the downward
// relation (2m+1) F_m = 2T F_{m+1} + exp(-T).
__device__ __forceinline__ void boys_scaled(const double* __restrict__ tab, const double* __restrict__ mid,
                                            double cL, int hi, int lo, double T, double pref, double* v,
                                            int stride) {
  double FL, ex;
  boys_top(tab, mid, cL, hi, hi > lo, T, FL, ex);  // exp(-T) only feeds the downward relation
  double G = pref * FL;
  v[(hi - lo) * stride] = G;
  if (hi > lo) {
    const double E = pref * ex, T2 = T + T;
    for (int m = hi - 1; m >= lo; --m) {
      G = fma(T2, G, E) * c_inv2m1[m];
      v[(m - lo) * stride] = G;
    }
  }
}

// ---------------------------------------------------------------------------
// precompute kernels
// ---------------------------------------------------------------------------


// One thread per primitive pair (pair p, a-primitive ia, b-primitive ib).
__device__ __forceinline__ void pair_record(const DevBasis& orb, const int32_t* __restrict__ pairs, int Ka, int Kb,
                                            double* __restrict__ rec, double* __restrict__ ab, long long i) {
  long long p = i / (Ka * Kb);
  int r = (int)(i - p * Ka * Kb);
  int ia = r / Kb, ib = r - ia * Kb;
  int sa = pairs[2 * p], sb = pairs[2 * p + 1];
  const double* A = orb.xyz + 3 * sa;
  const double* B = orb.xyz + 3 * sb;
  double za = orb.exps[orb.off[sa] + ia], ca = orb.coefs[orb.off[sa] + ia];
  double zb = orb.exps[orb.off[sb] + ib], cb = orb.coefs[orb.off[sb] + ib];
  double g = za + zb, ig = 1.0 / g;
  double AB[3] = {A[0] - B[0], A[1] - B[1], A[2] - B[2]};
  double ab2 = AB[0] * AB[0] + AB[1] * AB[1] + AB[2] * AB[2];
  const double two_pi52 = 34.98683665524972;  // 2 pi^{5/2}
  double* o = rec + i * kPairRec;
  o[PR_G] = g;
  o[PR_K] = ca * cb * exp(-za * zb * ig * ab2) * two_pi52 * ig;
  for (int x = 0; x < 3; ++x) {
    double P = (za * A[x] + zb * B[x]) * ig;
    o[PR_P + x] = P;
    o[PR_PA + x] = P - A[x];
  }
  for (int x = 0; x < 3; ++x) o[PR_PB + x] = o[PR_P + x] - B[x];
  o[PR_ZA] = za;
  o[PR_ZB] = zb;
  for (int nn = 1; nn <= 14; ++nn) o[PR_NH + nn - 1] = 0.5 * nn * ig;
  if (r == 0)
    for (int x = 0; x < 3; ++x) ab[3 * p + x] = AB[x];
}

// One thread per (ket list entry q, primitive ic): zeta_c and c_c / zeta_c.
__device__ __forceinline__ void aux_record(const DevBasis& aux, const int32_t* __restrict__ auxs, int Kc,
                                           double* __restrict__ rec, double* __restrict__ cxyz, long long i) {
  long long q = i / Kc;
  int ic = (int)(i - q * Kc);
  int s = auxs[q];
  double z = aux.exps[aux.off[s] + ic], c = aux.coefs[aux.off[s] + ic];
  rec[i * kAuxRec + 0] = z;
  rec[i * kAuxRec + 1] = c / z;
  if (ic == 0)
    for (int x = 0; x < 3; ++x) cxyz[3 * q + x] = aux.xyz[3 * s + x];
}

// Pair records by the first threads, ket records by the others (one launch:
// a small call is mostly launches).
__global__ void precompute_kernel(DevBasis orb, const int32_t* __restrict__ pairs, long long npair, int Ka, int Kb,
                                  double* __restrict__ rec, double* __restrict__ ab, DevBasis aux,
                                  const int32_t* __restrict__ auxs, long long naux, int Kc,
                                  double* __restrict__ auxrec, double* __restrict__ auxc) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x, n = npair * Ka * Kb;
  if (i < n)
    pair_record(orb, pairs, Ka, Kb, rec, ab, i);
  else if (i - n < naux * Kc)
    aux_record(aux, auxs, Kc, auxrec, auxc, i - n);
}

// The same for many lists in one launch (a DF-J build has dozens of groups, and
// a launch each of a few microseconds came to 0.6 of 22.3 ms for eight densities
// on 16 atoms).  Each warp finds its block's job among the first blocks.
__global__ void precompute_jobs_kernel(DevBasis orb, DevBasis aux, const PrecomputeJob* __restrict__ jobs, int n) {
  const int lane = threadIdx.x & 31;
  int at = 0;
  for (int b = 0; b < n; b += 32)
    at += __popc(__ballot_sync(0xffffffffu, b + lane < n && jobs[b + lane].first <= (long long)blockIdx.x));
  const PrecomputeJob& j = jobs[at - 1];
  const long long i = (blockIdx.x - j.first) * blockDim.x + threadIdx.x, np = j.npair * j.Ka * j.Kb;
  if (i < np)
    pair_record(orb, j.pairs, j.Ka, j.Kb, j.rec, j.ab, i);
  else if (i - np < j.naux * j.Kc)
    aux_record(aux, j.auxs, j.Kc, j.auxrec, j.auxc, i - np);
}

// ---------------------------------------------------------------------------
// integral kernel
// ---------------------------------------------------------------------------

#define BUF_T(b, idx, t) ((b).base + (idx) * (b).si + (t) * (b).st)
#define BUF_TG(b, idx, g, t) ((b).base + (idx) * (b).si + (g) * (b).sg + (t) * (b).st)

// item w -> (t, x) for per-triple stages with X targets
__device__ __forceinline__ void dec2(unsigned w, int mode, const FDiv& fT, const FDiv& fX, int& t, int& x) {
  if (mode == 0) {
    unsigned q = fT.div(w);
    t = (int)(w - q * fT.d);
    x = (int)q;
  } else {
    unsigned q = fX.div(w);
    x = (int)(w - q * fX.d);
    t = (int)q;
  }
}

// item w -> (t, g, x) for per-(triple, primitive) stages
__device__ __forceinline__ void dec3(unsigned w, int mode, const FDiv& fT, const FDiv& fG, const FDiv& fX, int& t,
                                     int& g, int& x) {
  if (mode == 0) {
    unsigned q = fT.div(w);
    t = (int)(w - q * fT.d);
    unsigned r = fG.div(q);
    g = (int)(q - r * fG.d);
    x = (int)r;
  } else {
    unsigned q = fX.div(w);
    x = (int)(w - q * fX.d);
    unsigned r = fG.div(q);
    g = (int)(q - r * fG.d);
    t = (int)r;
  }
}

// A stage's loop over nx targets of T triples in blocks of TB: f(x, t0, ts)
// for the triples t0, t0 + ts, ..., TB of them (those at or beyond the tile's
// count are the caller's to skip).  Lanes run over triples first (mode 0) or
// targets first (mode 1).
template <int NT, int TB, class F>
__device__ __forceinline__ void stage_items(int nx, int T, int tv, int mode, const F& f) {
  FDiv fd;
  const int nt = T / TB;
  fd.init(mode == 0 ? nt : nx);
  for (unsigned w = threadIdx.x; w < (unsigned)(nt * nx); w += NT) {
    const unsigned q = fd.div(w), r = w - q * fd.d;
    if (mode == 0) {
      if ((int)r < tv) f((int)q, (int)r, nt);
    } else {
      if ((int)q * TB < tv) f((int)r, (int)q * TB, 1);
    }
  }
}

// Blocks of four, two or one triples, as T divides, as long as the items still
// fill the block's threads and (mode 0) a warp holds two targets at most.
template <int NT, class F>
__device__ __forceinline__ void stage(int nx, int T, int tv, int mode, const F& f) {
  const int most = mode == 0 ? T >> 4 : 4;
  if ((T & 3) == 0 && most >= 4 && nx * T >= 4 * NT)
    stage_items<NT, 4>(nx, T, tv, mode, [&](int x, int t0, int ts) { f(x, t0, ts, Int<4>()); });
  else if ((T & 1) == 0 && most >= 2 && nx * T >= 2 * NT)
    stage_items<NT, 2>(nx, T, tv, mode, [&](int x, int t0, int ts) { f(x, t0, ts, Int<2>()); });
  else
    stage_items<NT, 1>(nx, T, tv, mode, [&](int x, int t0, int ts) { f(x, t0, ts, Int<1>()); });
}

// Segmented dot products out[o] += sum_{r < len} prod(o, r) for o < nout,
// each partial result handed to emit(o, value), which adds it to global
// memory with an atomic.  The FP64 pipe charges a whole warp instruction
// whatever the number of active lanes, and one lane's dependent FMAs are
// serialised, so the mapping follows the estimated chain length: one lane per
// output (two partial sums) when there are many outputs, else one warp per
// (output, 128-term chunk) whose lanes each emit their own partial sum (a warp
// shuffle reduction here costs the whole kernel registers).
template <int NT, class Prod, class Emit>
__device__ __forceinline__ void seg_dot(int nout, int len, const Prod& prod, const Emit& emit) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kWarps = NT / 32, kChunk = 128;
  if (nout <= 0 || len <= 0) return;
  const int nch = (len + kChunk - 1) / kChunk;
  const long long lane_steps = (long long)((nout + NT - 1) / NT) * ((len + 1) / 2);
  const long long warp_steps = (long long)((nout * nch + kWarps - 1) / kWarps) * ((min(len, kChunk) + 31) / 32 + 1);
  if (lane_steps <= warp_steps) {
    for (int o = tid; o < nout; o += NT) {
      double s0 = 0.0, s1 = 0.0;
      int r = 0;
      for (; r + 1 < len; r += 2) {
        s0 = prod(o, r, s0);
        s1 = prod(o, r + 1, s1);
      }
      if (r < len) s0 = prod(o, r, s0);
      emit(o, s0 + s1);
    }
  } else {
    for (int it = warp; it < nout * nch; it += kWarps) {
      const int o = it / nch, r0 = (it - o * nch) * kChunk, r1 = min(len, r0 + kChunk);
      if (r0 + lane >= r1) continue;
      double s = 0.0;
      for (int r = r0 + lane; r < r1; r += 32) s = prod(o, r, s);
      emit(o, s);
    }
  }
}

// HRR rounds (Eq. hrr; Sec. 2.5.5 for two-quantum rounds) and the optional
// solid-harmonic bra transforms on tv triples of H[0]; returns the buffer
// holding the final block.
template <int NT>
__device__ __forceinline__ Buf hrr_and_bra(const ClassDesc& d, double* sm, int T, int tv, int mode) {
  // ---- HRR (Eq. hrr) round by round: each row is dst = sum_t coef_t src_t
  // over 2 terms (one quantum moved, Eq. hrr) or 3-4 terms (two quanta,
  // Sec. 2.5.5), the coefficients products of AB components
  FDiv fC;
  fC.init(d.nC);
  for (int j = 1; j <= d.nhrr; ++j) {
    const Buf hi = d.H[j - 1], ho = d.H[j];
    const double* abp = sm + d.ab_base;
    const uint4* tab = d.htab + d.hstart[j];
    const int nC = d.nC;
    stage<NT>(d.hrows[j] * nC, T, tv, mode, [&](int x, int t0, int ts, auto tb) {
      constexpr int TB = decltype(tb)::n;
      const int r = (int)fC.div(x), C = x - r * nC;
      const uint4 e = __ldg(tab + r);
      const unsigned nt = e.x >> 16;
      const int st = hi.st * ts, base = hi.base + t0 * hi.st + C * hi.si, row = nC * hi.si;
      const double* s0 = sm + base + (int)(e.y & 0xFFFF) * row;
      const double* s1 = sm + base + (int)(e.y >> 16) * row;
      double* o = sm + BUF_T(ho, (int)(e.x & 0xFFFF) * nC + C, t0);
      const int so = ho.st * ts;
      const double c1 = abp[(e.w >> 4) & 0xF];
      double v[TB];
#pragma unroll
      for (int k = 0; k < TB; ++k)
        if (t0 + k * ts < tv) v[k] = fma(c1, s1[k * st], s0[k * st]);
      if (nt > 2) {
        const double* s2 = sm + base + (int)(e.z & 0xFFFF) * row;
        const double c2 = abp[(e.w >> 8) & 0xF];
#pragma unroll
        for (int k = 0; k < TB; ++k)
          if (t0 + k * ts < tv) v[k] = fma(c2, s2[k * st], v[k]);
        if (nt > 3) {
          const double* s3 = sm + base + (int)(e.z >> 16) * row;
          const double c3 = abp[(e.w >> 12) & 0xF];
#pragma unroll
          for (int k = 0; k < TB; ++k)
            if (t0 + k * ts < tv) v[k] = fma(c3, s3[k * st], v[k]);
        }
      }
#pragma unroll
      for (int k = 0; k < TB; ++k)
        if (t0 + k * ts < tv) o[k * so] = v[k];
    });
    __syncthreads();
  }
  // ---- optional solid-harmonic bra
  Buf cur = d.H[d.nhrr];
  // out[dst] = sum of coef[q] src[entry q] over the CSR row [q0, q1); a single
  // unit coefficient is a copy
  const auto row_sum = [&](const int2* ent, int q0, int q1, const Buf& in, int in0, int stride, const Buf& out, int dst,
                           int t0, int ts, auto tb) {
    constexpr int TB = decltype(tb)::n;
    const int st = in.st * ts, so = out.st * ts;
    const double* src = sm + in.base + t0 * in.st + in0 * in.si;
    double* o = sm + BUF_T(out, dst, t0);
    double v[TB];
    const int2 e0 = __ldg(ent + q0);
    const double* p0 = src + e0.x * stride * in.si;
    if (e0.y == 0) {
#pragma unroll
      for (int k = 0; k < TB; ++k) v[k] = t0 + k * ts < tv ? p0[k * st] : 0.0;
    } else {
      const double c = __ldg(d.pal + e0.y);
#pragma unroll
      for (int k = 0; k < TB; ++k)
        if (t0 + k * ts < tv) v[k] = c * p0[k * st];
    }
    for (int q = q0 + 1; q < q1; ++q) {
      const int2 e = __ldg(ent + q);
      const double* p = src + e.x * stride * in.si;
      const double c = __ldg(d.pal + e.y);
#pragma unroll
      for (int k = 0; k < TB; ++k)
        if (t0 + k * ts < tv) v[k] = fma(c, p[k * st], v[k]);
    }
#pragma unroll
    for (int k = 0; k < TB; ++k)
      if (t0 + k * ts < tv) o[k * so] = v[k];
  };
  if (d.nbA) {
    // items A-slowest: with targets across lanes they share A's trip count
    const int nB = d.ncB * d.nC;
    FDiv fB;
    fB.init(nB);
    stage<NT>(d.nbA * d.nC, T, tv, mode, [&](int x, int t0, int ts, auto tb) {
      const int A = (int)fB.div(x), bC = x - A * nB;
      row_sum(d.baent, __ldg(d.baptr + A), __ldg(d.baptr + A + 1), cur, bC, nB, d.BA, x, t0, ts, tb);
    });
    __syncthreads();
    cur = d.BA;
  }
  if (d.nbB) {
    // items B-slowest: with targets across lanes they share B's trip count
    const int nBs = d.nB, nAC = (d.nbB / d.nB) * d.nC, nC = d.nC;
    FDiv fAC;
    fAC.init(nAC);
    stage<NT>(d.nbB * nC, T, tv, mode, [&](int x, int t0, int ts, auto tb) {
      const int B = (int)fAC.div(x), rem = x - B * nAC;
      const int A = (int)fC.div(rem), C = rem - A * nC;
      row_sum(d.bbent, __ldg(d.bbptr + B), __ldg(d.bbptr + B + 1), cur, A * d.ncB * nC + C, nC, d.BB,
              (A * nBs + B) * nC + C, t0, ts, tb);
    });
    __syncthreads();
    cur = d.BB;
  }
  return cur;
}

// One tile: (sub-pair, up to T ket shells) through every stage, ending in the
// store or the DF-J digestion.  kVar selects the instantiation: 0 the plain
// kernel (store, per-integral DF-J digestion), 1 adds the several-density
// digestion on FP64 tensor-core tiles (digest == 4), in a kernel of its own
// so that the plain launches keep their register count.
template <int kVar, int NT>
__device__ __forceinline__ void tile_body(const ClassDesc& d, long long tile, double* sm) {
  const unsigned tid = threadIdx.x;
  const int T = d.T, G = d.G, mode = d.mode, lc = d.lc, Lab = d.Lab;
  FDiv fT, fG, fKc;
  fT.init(T);
  fG.init(G);
  fKc.init(d.Kc);
  const int auxsz = 3 + kAuxRec * d.Kc;
  {
    long long sub;
    int aux0, tv;
    if (d.tiles) {
      const int4 tt = __ldg(d.tiles + tile);
      sub = tt.x;
      aux0 = tt.y;
      tv = tt.z;
    } else {
      sub = tile / d.ntile_aux;
      aux0 = (int)(tile - sub * d.ntile_aux) * T;
      tv = (int)min((long long)T, d.naux - aux0);
    }
    const int4 sp = __ldg(d.subpairs + sub);
    const long long pair = sp.x;
    const int kab = sp.z, accum = sp.w;
    if (kab == 0) {  // (uniform across the CTA)
      // a sub-pair without primitive pairs adds nothing; its blocks are zero
      // when the pair has no other sub-pair
      if (accum == 2 && d.digest == 0) {
        double* o = d.out + ((pair - d.out_pair0) * d.naux + aux0) * (long long)d.nblk;
        for (int w = tid; w < tv * d.nblk; w += NT) o[w] = 0.0;
      }
      return;
    }
    const int K = kab * d.Kc;
    const int nchunk = (K + G - 1) / G;
    __syncthreads();  // previous tile done with shared memory
    {
      // this sub-pair's primitive-pair records, in its orientation
      for (int i = tid; i < kab * kPairRec; i += NT) {
        const int g = i / kPairRec, f = i - g * kPairRec;
        int fs = f;
        if (d.orient) {
          if (f >= PR_PA && f < PR_PA + 3) fs = f + (PR_PB - PR_PA);
          else if (f == PR_ZA) fs = PR_ZB;
          else if (f == PR_ZB) fs = PR_ZA;
        }
        const long long r = pair * d.Kab_rec + __ldg(d.primidx + sp.y + g);
        sm[d.pair_base + i] = d.pairrec[r * kPairRec + fs];
      }
      if (tid < 13) {
        // the HRR coefficients: 1, AB_i, 2 AB_i, AB_i^2, AB_x AB_y, AB_x AB_z, AB_y AB_z
        const double sg = d.orient ? -1.0 : 1.0;
        const double x = sg * d.pairab[pair * 3], y = sg * d.pairab[pair * 3 + 1], z = sg * d.pairab[pair * 3 + 2];
        const int ax = tid >= 1 && tid <= 9 ? (int)(tid - 1) % 3 : 0;
        const double u = ax == 0 ? x : (ax == 1 ? y : z);
        double v = 1.0;
        if (tid >= 1 && tid <= 3) v = u;
        else if (tid >= 4 && tid <= 6) v = 2.0 * u;
        else if (tid >= 7 && tid <= 9) v = u * u;
        else if (tid == 10) v = x * y;
        else if (tid == 11) v = x * z;
        else if (tid == 12) v = y * z;
        sm[d.ab_base + tid] = v;
      }
      for (int i = tid; i < tv * auxsz; i += NT) {
        int t = i / auxsz, r = i - t * auxsz;
        sm[d.aux_base + i] = r < 3 ? d.auxc[(long long)(aux0 + t) * 3 + r]
                                   : d.auxrec[(long long)(aux0 + t) * d.Kc * kAuxRec + (r - 3)];
      }
    }
    __syncthreads();

    for (int chunk = 0; chunk < nchunk; ++chunk) {
      const int p0 = chunk * G;
      const int gcnt = min(G, K - p0);
      // ---- stage A: geometry, Boys function, [00|0]^(m) and recurrence factors
      for (unsigned w = tid; w < (unsigned)(T * G); w += NT) {
        int t, g;
        if (mode == 0) {
          unsigned q = fT.div(w);
          t = (int)(w - q * T);
          g = (int)q;
        } else {
          unsigned q = fG.div(w);
          g = (int)(w - q * G);
          t = (int)q;
        }
        if (t >= tv || g >= gcnt) continue;
        const int p = p0 + g;
        const int ip = (int)fKc.div(p), ic = p - ip * d.Kc;
        const double* pr = sm + d.pair_base + ip * kPairRec;
        const double* ax = sm + d.aux_base + t * auxsz;
        const double gam = pr[PR_G], zc = ax[3 + kAuxRec * ic], ccp = ax[4 + kAuxRec * ic];
        const double s = gam + zc;
        const double rs = rsqrt_fp64(s);
        const double r = rs * rs;
        const double rg = zc * r;    // rho / gamma
        const double gr = gam * r;   // rho / zeta_c
        const double PCx = pr[PR_P] - ax[0], PCy = pr[PR_P + 1] - ax[1], PCz = pr[PR_P + 2] - ax[2];
        const double pc2 = fma(PCz, PCz, fma(PCy, PCy, PCx * PCx));
        const double rho = gam * rg;
        const double Tb = rho * pc2;
        const double pref = pr[PR_K] * ccp * rs;
        const int fb = BUF_TG(d.F, 0, g, t);
        const int fs = d.F.si;
        if (Lab > 0) {  // VRR1 factors (rho/gamma) PC
          sm[fb] = rg * PCx;
          sm[fb + fs] = rg * PCy;
          sm[fb + 2 * fs] = rg * PCz;
        }
        sm[fb + 3 * fs] = rg;
        if (lc > 0) {
          sm[fb + 4 * fs] = gr * PCx;
          sm[fb + 5 * fs] = gr * PCy;
          sm[fb + 6 * fs] = gr * PCz;
          const double Y = 0.5 * r;
          double v = Y;
          for (int k = 1; k <= d.kmax; ++k) {
            sm[fb + (6 + k) * fs] = v;
            v *= Y;
          }
        }
        boys_scaled(d.boys_tab, d.boys_mid, d.boys_cL, d.L, lc, Tb, pref, sm + BUF_TG(d.V, 0, g, t), d.V.si);
      }
      __syncthreads();
      // ---- weights W_{k,m} = Y^k s_{lc-k,m}(X), one item per (slot, |m|);
      // items of one m stand together (the loops' trip counts depend on it),
      // and the last threads take them, as the first VRR1 level starts on the
      // first
      {
        FDiv fS;
        const int ns = T * G, kmax = d.kmax;
        fS.init(ns);
        for (unsigned w = NT - 1 - tid; w < (unsigned)(ns * (lc + 1)); w += NT) {
          const int m = (int)fS.div(w), slot = (int)w - m * ns;
          int t, g;
          if (mode == 0) {
            g = (int)fT.div(slot);
            t = slot - g * T;
          } else {
            t = (int)fG.div(slot);
            g = slot - t * G;
          }
          if (t >= tv || g >= gcnt) continue;
          const double* F = sm + BUF_TG(d.F, 0, g, t);
          double* W = sm + BUF_TG(d.W, 0, g, t);
          const int fs = d.F.si, ws = d.W.si;
          if (lc == 0) {
            W[0] = 1.0;
            continue;
          }
          harmonic_weights(
              lc, kmax, m, F[4 * fs], F[5 * fs], F[6 * fs], c_q, [&](int k) { return F[(6 + k) * fs]; },
              [&](int i, double v) { W[i * ws] = v; });
        }
      }
      // ---- VRR1, level by level (Eq. vrr1).  A level is few targets and a
      // barrier: with few triples every (target, primitive, triple) is an item
      // of its own, with 16 or more an item is its target over the chunk's
      // primitives ((dd|f) K = 3: 6.4 -> 6.1 ms; one triple: 93 -> 102 ms)
      for (int e = 1; e <= Lab; ++e) {
        const int j0 = d.vlev_start[e - 1];
        const int nl = d.vlev_start[e] - j0, vs = d.V.si, fs = d.F.si;
        const auto target = [&](const uint4& it, int axis, int nq, double pa, double nh, int g, int t) {
          double* v = sm + BUF_TG(d.V, 0, g, t);
          const double* f = sm + BUF_TG(d.F, 0, g, t);
          double val = pa * v[(it.x >> 16) * vs];
          val = fma(-f[axis * fs], v[(it.y & 0xFFFF) * vs], val);
          if (nq) val = fma(nh, fma(-f[3 * fs], v[(it.z & 0xFFFF) * vs], v[(it.y >> 16) * vs]), val);
          v[(it.x & 0xFFFF) * vs] = val;
        };
        if (T >= 16) {
          stage<NT>(nl, T, tv, mode, [&](int x, int t0, int ts, auto tb) {
            constexpr int TB = decltype(tb)::n;
            const uint4 it = __ldg(d.vtab + j0 + x);
            const int axis = (it.z >> 16) & 0xF, nq = (it.z >> 20) & 0xF;
            for (int g = 0; g < gcnt; ++g) {
              const double* pr = sm + d.pair_base + (int)fKc.div(p0 + g) * kPairRec;
              const double pa = pr[PR_PA + axis], nh = nq ? pr[PR_NH + nq - 1] : 0.0;
#pragma unroll
              for (int k = 0; k < TB; ++k)
                if (t0 + k * ts < tv) target(it, axis, nq, pa, nh, g, t0 + k * ts);
            }
          });
        } else {
          FDiv fX;
          fX.init(nl);
          for (unsigned w = tid; w < (unsigned)(T * G * nl); w += NT) {
            int t, g, x;
            dec3(w, mode, fT, fG, fX, t, g, x);
            if (t >= tv || g >= gcnt) continue;
            const uint4 it = __ldg(d.vtab + j0 + x);
            const int axis = (it.z >> 16) & 0xF, nq = (it.z >> 20) & 0xF;
            const double* pr = sm + d.pair_base + (int)fKc.div(p0 + g) * kPairRec;
            target(it, axis, nq, pr[PR_PA + axis], nq ? pr[PR_NH + nq - 1] : 0.0, g, t);
          }
        }
        __syncthreads();
      }
      if (Lab == 0) __syncthreads();
      // ---- accumulate CVRR2 prerequisites over the chunk's primitives
      {
        const int vg = d.V.sg, wg = d.W.sg;
        stage<NT>(d.NACC, T, tv, mode, [&](int x, int t0, int ts, auto tb) {
          constexpr int TB = decltype(tb)::n;
          const unsigned e = __ldg(d.atab + x);
          const double* v = sm + BUF_TG(d.V, (int)(e & 0xFFFF), 0, t0);
          const double* w = sm + BUF_TG(d.W, (int)(e >> 16), 0, t0);
          double* p = sm + BUF_T(d.P, x, t0);
          const int sv = d.V.st * ts, sw = d.W.st * ts, sp_ = d.P.st * ts;
          double acc[TB];
          const bool full = t0 + (TB - 1) * ts < tv;
#pragma unroll
          for (int k = 0; k < TB; ++k) acc[k] = (full || t0 + k * ts < tv) ? (chunk ? p[k * sp_] : 0.0) : 0.0;
          if (full) {
#pragma unroll 2
            for (int g = 0; g < gcnt; ++g)
#pragma unroll
              for (int k = 0; k < TB; ++k) acc[k] = fma(v[k * sv + g * vg], w[k * sw + g * wg], acc[k]);
#pragma unroll
            for (int k = 0; k < TB; ++k) p[k * sp_] = acc[k];
          } else {
#pragma unroll
            for (int k = 0; k < TB; ++k)
              if (t0 + k * ts < tv) {
                for (int g = 0; g < gcnt; ++g) acc[k] = fma(v[k * sv + g * vg], w[k * sw + g * wg], acc[k]);
                p[k * sp_] = acc[k];
              }
          }
        });
      }
      __syncthreads();
    }

    // ---- CVRR2 targets (a 0|C) by the n-quantum gather (Sec. 2.5.4), the ket
    // already solid harmonic
    if (d.comp) {
      FDiv fX;
      fX.init(d.ngt);
      for (unsigned w = tid; w < (unsigned)(T * d.ngt); w += NT) {
        int t, r;
        dec2(w, mode, fT, fX, t, r);
        if (t >= tv) continue;
        const int id = __ldg(d.gdst + r);
        Dot2 acc;
        for (int q = __ldg(d.gptr + id); q < __ldg(d.gptr + id + 1); ++q) {
          const unsigned e = __ldg(d.gterm + q);
          acc.add(__ldg(d.pal + (e >> kGatherBits)), sm[BUF_T(d.P, e & kGatherMask, t)]);
        }
        sm[BUF_T(d.H[0], id, t)] = acc.value();
      }
    } else {
      // lanes that share the target (mode 0) walk its CSR row by broadcast
      // loads; lanes on consecutive targets (mode 1; the list padded to whole
      // warps) a sliced-ELL copy, one coalesced line per term step and one trip
      // count per slice
      stage<NT>(mode == 0 ? d.ngt : (d.ngt + 31) & ~31, T, tv, mode, [&](int r, int t0, int ts, auto tb) {
        constexpr int TB = decltype(tb)::n;
        if (r >= d.ngt) return;
        const int id = __ldg(d.gdst + r);
        const unsigned* ge;
        int n, step;
        if (mode == 0) {
          const int q0 = __ldg(d.gptr + id);
          ge = d.gterm + q0;
          n = __ldg(d.gptr + id + 1) - q0;
          step = 1;
        } else {
          const int2 sl = __ldg(d.gslice + (r >> 5));
          ge = d.gell + sl.x + (r & 31);
          n = sl.y;
          step = 32;
        }
        const double* P = sm + d.P.base + t0 * d.P.st;
        const int st = d.P.st * ts, si = d.P.si;
        double s[TB];
#pragma unroll
        for (int k = 0; k < TB; ++k) s[k] = 0.0;
        const bool full = t0 + (TB - 1) * ts < tv;
        if (full) {
#pragma unroll 2
          for (int j = 0; j < n; ++j) {
            const unsigned e = __ldg(ge + j * step);
            const double c = __ldg(d.pal + (e >> kGatherBits));
            const double* p = P + (int)(e & kGatherMask) * si;
#pragma unroll
            for (int k = 0; k < TB; ++k) s[k] = fma(c, p[k * st], s[k]);
          }
        } else {
          for (int j = 0; j < n; ++j) {
            const unsigned e = __ldg(ge + j * step);
            const double c = __ldg(d.pal + (e >> kGatherBits));
            const double* p = P + (int)(e & kGatherMask) * si;
#pragma unroll
            for (int k = 0; k < TB; ++k)
              if (t0 + k * ts < tv) s[k] = fma(c, p[k * st], s[k]);
          }
        }
#pragma unroll
        for (int k = 0; k < TB; ++k)
          if (t0 + k * ts < tv) sm[BUF_T(d.H[0], id, t0 + k * ts)] = s[k];
      });
    }
    __syncthreads();
    Buf cur = hrr_and_bra<NT>(d, sm, T, tv, mode);
    if (d.digest == 3) {
      // ---- matrix store (2-centre metric (P|Q) = (P 1|Q), nB = 1): element
      // (t, A, C) of the tile goes to out[(ao_pair + A) * ldD + ao_ket + C]
      const int4 pao = __ldg(d.pair_ao + pair);
      const int nA = d.onA, nC = d.nC, nAC = nA * nC;
      FDiv fAC, fC;
      fAC.init(nAC);
      fC.init(nC);
      const unsigned n = (unsigned)(tv * nAC);
      for (unsigned w = tid; w < n; w += NT) {
        const int t = (int)fAC.div(w), r = (int)(w - (unsigned)t * nAC);
        const int A = (int)fC.div(r), C = r - A * nC;
        d.out[(long long)(pao.x + A) * d.ldD + __ldg(d.aux_ao + aux0 + t) + C] = sm[BUF_T(cur, A * nC + C, t)];
      }
      return;
    }
    if (kVar == 1 && d.digest == 4) {
      // ---- DF-J digestion for nd <= 8 densities at once, as two small GEMMs
      // on FP64 tensor-core tiles (m8n8k4), with M rows per warp tile:
      //   gamma[d][t][C] = wg * sum_s I[t][s][C] Ds[s][d]    (M = tv*nC, K = nAB)
      //   J[d][s]        = wj * sum_{t,C} I[t][s][C] Cs[t*nC+C][d]  (M = nAB, K = tv*nC)
      const int4 pao = __ldg(d.pair_ao + pair);
      const double wg = pao.z ? 1.0 : 2.0, wj = pao.z ? 0.5 : 1.0;
      const int nA = d.onA, nB = d.onB, nC = d.nC, nAB = nA * nB, R = tv * nC, nd = d.nd;
      const int kAB = (nAB + 3) & ~3, kR = (R + 3) & ~3;
      double* Ds = sm + d.dscr;      // [kAB][8]
      double* Cs = Ds + kAB * 8;     // [kR][8]
      for (int i = tid; i < kAB * 8; i += NT) {
        const int r = i >> 3, dd = i & 7;  // r: storage index of (A, B)
        const int A = d.orient ? r % nA : r / nB, B = d.orient ? r / nA : r % nB;
        Ds[i] = (d.gamma && r < nAB && dd < nd)
                    ? __ldg(d.D + dd * d.dstride + (long long)(pao.x + A) * d.ldD + pao.y + B)
                    : 0.0;
      }
      for (int i = tid; i < kR * 8; i += NT) {
        const int r = i >> 3, dd = i & 7;
        double v = 0.0;
        if (d.J && r < R && dd < nd) {
          const int t = r / nC, C = r - t * nC;
          v = __ldg(d.cvec + dd * d.cstride + __ldg(d.aux_ao + aux0 + t) + C);
        }
        Cs[i] = v;
      }
      __syncthreads();
      const Buf cb = cur;
      const int lane = tid & 31, warp = tid >> 5, g = lane >> 2, q = lane & 3;
      constexpr int kWarps = NT / 32;
      if (d.gamma) {
        for (int m0 = warp * 8; m0 < R; m0 += kWarps * 8) {
          const int m = m0 + g;
          const int t = m / nC, C = m - t * nC;
          double c0 = 0.0, c1 = 0.0;
          for (int k0 = 0; k0 < kAB; k0 += 4) {
            const int k = k0 + q;
            const double a = (m < R && k < nAB) ? sm[BUF_T(cb, k * nC + C, t)] : 0.0;
            dmma_8x8x4(a, Ds[(k0 + q) * 8 + g], c0, c1);
          }
          if (m < R) {
            double* gm = d.gamma + __ldg(d.aux_ao + aux0 + t) + C;
            if (2 * q < nd) atomicAdd(gm + (2 * q) * d.cstride, wg * c0);
            if (2 * q + 1 < nd) atomicAdd(gm + (2 * q + 1) * d.cstride, wg * c1);
          }
        }
      }
      if (d.J) {
        for (int m0 = warp * 8; m0 < nAB; m0 += kWarps * 8) {
          const int m = m0 + g;  // storage index s of the block
          double c0 = 0.0, c1 = 0.0;
          for (int k0 = 0; k0 < kR; k0 += 4) {
            const int k = k0 + q;
            const int t = k / nC, C = k - t * nC;
            const double a = (m < nAB && k < R) ? sm[BUF_T(cb, m * nC + C, t)] : 0.0;
            dmma_8x8x4(a, Cs[(k0 + q) * 8 + g], c0, c1);
          }
          if (m < nAB) {
            const int A = d.orient ? m % nA : m / nB, B = d.orient ? m / nA : m % nB;
            double* Jm = d.J + (long long)(pao.x + A) * d.ldD + pao.y + B;
            if (2 * q < nd) atomicAdd(Jm + (2 * q) * d.dstride, wj * c0);
            if (2 * q + 1 < nd) atomicAdd(Jm + (2 * q + 1) * d.dstride, wj * c1);
          }
        }
      }
      return;
    }
    if (d.digest) {
      // ---- DF-J digestion (Sec. 3): the block never leaves shared memory.
      // With s the block's (A, B) index in its storage order:
      //   gamma[t][C] = wg * sum_s I[t][s][C] Ds[s]        (Ds = D block)
      //   J[s]        = wj * sum_{t,C} I[t][s][C] Cs[t][C]  (Cs = c of the tile's kets)
      const int4 pao = __ldg(d.pair_ao + pair);
      const double wg = pao.z ? 1.0 : 2.0, wj = pao.z ? 0.5 : 1.0;
      const int nA = d.onA, nB = d.onB, nC = d.nC, nAB = nA * nB;
      double* Ds = sm + d.dscr;
      double* Cs = Ds + nAB;
      const int sA = d.orient ? 1 : nB, sB = d.orient ? nA : 1;  // storage index of (A, B)
      if (d.gacc)
        for (int s = tid; s < nAB; s += NT) {
          const int A = s / nB, B = s - A * nB;
          Ds[A * sA + B * sB] = __ldg(d.D + (long long)(pao.x + A) * d.ldD + pao.y + B);
        }
      if (d.Jacc)
        for (int i = tid; i < tv * nC; i += NT) {
          const int t = i / nC, C = i - t * nC;
          Cs[i] = __ldg(d.cvec + __ldg(d.aux_ao + aux0 + t) + C);
        }
      __syncthreads();
      const Buf cb = cur;
      FDiv fC;
      fC.init(nC);
      if (d.gacc)
        seg_dot<NT>(tv * nC, nAB,
                [&](int o, int r, double acc) {
                  const int t = (int)fC.div(o), C = o - t * nC;
                  return fma(sm[BUF_T(cb, r * nC + C, t)], Ds[r], acc);
                },
                [&](int o, double v) {
                  const int t = (int)fC.div(o), C = o - t * nC;
                  fix_add(d.gacc + kFixWords * (__ldg(d.aux_ao + aux0 + t) + C), wg * v);
                });
      if (d.Jacc)
        seg_dot<NT>(nAB, tv * nC,
                [&](int o, int r, double acc) {
                  const int t = (int)fC.div(r), C = r - t * nC;
                  return fma(sm[BUF_T(cb, o * nC + C, t)], Cs[r], acc);
                },
                [&](int o, double v) {
                  const int A = d.orient ? o % nA : o / nB, B = d.orient ? o / nA : o % nB;
                  fix_add(d.Jacc + kFixWords * ((long long)(pao.x + A) * d.ldD + pao.y + B), wj * v);
                });
      return;
    }
    // ---- store the tile's contiguous output block (transposed into the
    // caller's (A, B) order for B-oriented sub-pairs; added to the block
    // already written by the A-oriented launch when the pair has both)
    {
      FDiv fB, fBC, fC;
      fB.init(d.nblk);
      fBC.init(d.onB * d.nC);
      fC.init(d.nC);
      double* o = d.out + ((pair - d.out_pair0) * d.naux + aux0) * (long long)d.nblk;
      const unsigned n = (unsigned)(tv * d.nblk);
      for (unsigned w = tid; w < n; w += NT) {
        const unsigned t = fB.div(w);
        const int idx = (int)(w - t * d.nblk);
        int sidx = idx;
        if (d.orient) {
          const int A = (int)fBC.div(idx), rem = idx - A * d.onB * d.nC;
          const int B = (int)fC.div(rem), C = rem - B * d.nC;
          sidx = (B * d.onA + A) * d.nC + C;
        }
        double v = sm[BUF_T(cur, sidx, (int)t)];
        if (accum) v += o[w];
        o[w] = v;
      }
    }
  }
}

// One class launch: CTAs stride over the class's tiles.  384 threads and 56
// registers when three CTAs fit an SM's shared memory (their barriers overlap
// better: (ff|g) K = 1 12.5 -> 10.8 ms), else 512 threads and two CTAs ((gg|i)
// K = 6, one triple per tile, 99 -> 93 ms).  kVar 1: DF-J launches digesting
// several densities.
template <int kVar, int NT, int NB>
__global__ void __launch_bounds__(NT, NB) eri3c_kernel(const __grid_constant__ ClassDesc d) {
  extern __shared__ double sm[];
  for (long long tile = blockIdx.x; tile < d.ntiles; tile += gridDim.x) tile_body<kVar, NT>(d, tile, sm);
}

// Both orientations of a small plan (one tile per SM at most) side by side: the
// first ga CTAs take a's tiles, the others b's.
constexpr int kBothThreads = 512;
__global__ void __launch_bounds__(kBothThreads, 1) eri3c_kernel_both(const __grid_constant__ ClassDesc a,
                                                                     const __grid_constant__ ClassDesc b, int ga) {
  extern __shared__ double sm[];
  if ((int)blockIdx.x < ga) {
    for (long long tile = blockIdx.x; tile < a.ntiles; tile += ga) tile_body<0, kBothThreads>(a, tile, sm);
  } else {
    for (long long tile = blockIdx.x - ga; tile < b.ntiles; tile += gridDim.x - ga)
      tile_body<0, kBothThreads>(b, tile, sm);
  }
}

// (s s|C) classes (la = lb = 0) stored per integral, one thread per triple.
// With a = 0 the n-quantum CVRR2 has the single term u = 0, so the (0 0|c)
// target is the prerequisite P_c = sum over primitive triples of
// [00|0]^(lc) X^c (Eq. a0cv2, k = 0; X = (gamma / (gamma + zeta_c)) PC), the
// same quantities the tile kernel forms.  The NC accumulators live in
// registers and the primitive loop has no barrier; the ket transform runs
// from a shared-memory copy, and the block stores its triples' blocks
// element-major (coalesced when the triples' blocks are contiguous).
constexpr int kSsThreads = 128;

// Doubles from one lane's row of n to the next lane's: odd, so that the lanes
// fall on different banks (rows of 16 doubles, (s s|g) and (p s|g), put all 32
// on one: (p s|g) K = 1, 2048 x 512, 0.83 -> 0.58 ms, with one read of the
// ket table for the three bra components).
__host__ __device__ constexpr int odd_stride(int n) { return n | 1; }

// The primitive loop of one (s s|C) triple: acc[c] += [00|0]^(lc) X^c over
// the sub-pair's primitive pairs and the ket shell's primitives.
template <int LC>
__device__ __forceinline__ void ss_prims(const ClassDesc& d, long long pair, const int4& sp, long long q,
                                         double* acc) {
  const double Cx = __ldg(d.auxc + 3 * q), Cy = __ldg(d.auxc + 3 * q + 1), Cz = __ldg(d.auxc + 3 * q + 2);
  for (int ip = 0; ip < sp.z; ++ip) {
    const double* pr = d.pairrec + (pair * d.Kab_rec + __ldg(d.primidx + sp.y + ip)) * kPairRec;
    const double gam = __ldg(pr + PR_G), K = __ldg(pr + PR_K);
    const double PCx = __ldg(pr + PR_P) - Cx, PCy = __ldg(pr + PR_P + 1) - Cy, PCz = __ldg(pr + PR_P + 2) - Cz;
    const double pc2 = fma(PCz, PCz, fma(PCy, PCy, PCx * PCx));
    for (int ic = 0; ic < d.Kc; ++ic) {
      const double zc = __ldg(d.auxrec + (q * d.Kc + ic) * kAuxRec);
      const double ccp = __ldg(d.auxrec + (q * d.Kc + ic) * kAuxRec + 1);
      const double sg = gam + zc;
      const double rs = rsqrt_fp64(sg);
      const double r = rs * rs;
      const double gr = gam * r;
      const double Tb = gr * zc * pc2;
      double V;
      boys_scaled(d.boys_tab, d.boys_mid, d.boys_cL, LC, LC, Tb, K * ccp * rs, &V, 0);
      if (LC == 0) {
        acc[0] += V;
      } else {
        // powers of X = gr PC; the monomials X^c in the Cartesian order (x
        // descending, then y descending), one FMA per target
        double px[LC + 1], py[LC + 1], pz[LC + 1];
        px[0] = V; py[0] = 1.0; pz[0] = 1.0;
        const double Xx = gr * PCx, Xy = gr * PCy, Xz = gr * PCz;
#pragma unroll
        for (int j = 1; j <= LC; ++j) {
          px[j] = px[j - 1] * Xx;
          py[j] = py[j - 1] * Xy;
          pz[j] = pz[j - 1] * Xz;
        }
        int c = 0;
#pragma unroll
        for (int nx = LC; nx >= 0; --nx)
#pragma unroll
          for (int ny = LC - nx; ny >= 0; --ny) {
            acc[c] = fma(px[nx], py[ny] * pz[LC - nx - ny], acc[c]);
            ++c;
          }
      }
    }
  }
}

template <int LC>
__global__ void __launch_bounds__(kSsThreads) eri3c_ss_kernel(const __grid_constant__ ClassDesc d) {
  constexpr int NC = (LC + 1) * (LC + 2) / 2, NS = 2 * LC + 1;
  __shared__ double sP[kSsThreads * odd_stride(NC)];
  __shared__ double sO[kSsThreads * NS];
  __shared__ long long sOff[kSsThreads];
  __shared__ int sAcc[kSsThreads];
  const int tid = threadIdx.x;
  const long long ntri = d.nsub * d.naux;
  for (long long base = (long long)blockIdx.x * kSsThreads; base < ntri; base += (long long)gridDim.x * kSsThreads) {
    const long long w = base + tid;
    double acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = 0.0;
    long long off = -1;
    int accum = 0;
    if (w < ntri) {
      const long long sub = w / d.naux;
      const long long q = w - sub * d.naux;
      const int4 sp = __ldg(d.subpairs + sub);
      accum = sp.w == 1;
      off = (((long long)sp.x - d.out_pair0) * d.naux + q) * (long long)d.nblk;
      ss_prims<LC>(d, sp.x, sp, q, acc);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) sP[tid * odd_stride(NC) + c] = acc[c];
    sOff[tid] = off;
    sAcc[tid] = accum;
    __syncthreads();
    // ket transform: element-major over the block's triples
    for (int i = tid; i < kSsThreads * NS; i += kSsThreads) {
      const int t = i / NS, C = i - t * NS;
      double v = 0.0;
      for (int k = __ldg(d.kptr + C); k < __ldg(d.kptr + C + 1); ++k) {
        const int2 e = __ldg(d.kent + k);
        v = fma(__ldg(d.pal + e.y), sP[t * odd_stride(NC) + e.x], v);
      }
      sO[i] = v;
    }
    __syncthreads();
    for (int i = tid; i < kSsThreads * NS; i += kSsThreads) {
      const int t = i / NS, C = i - t * NS;
      const long long o = sOff[t];
      if (o < 0) continue;
      double v = sO[i];
      if (sAcc[t]) v += d.out[o + C];
      d.out[o + C] = v;
    }
    __syncthreads();
  }
}

// Sums js[k] over the W lanes of a tile for eight densities: while there are
// values left to share, each step hands half of them to the other half of the
// lanes (nine additions instead of 40 for W = 32); then adds w times each sum to
// its density's J element.
__device__ __forceinline__ void multi_j(const ClassDesc& d, double (&js)[8], int W, int t, bool store, double w,
                                        long long elem) {
  int first = 0, left = 8, o = W >> 1;
#pragma unroll
  for (int n = 4; n > 0; n >>= 1) {
    if (o > 0) {
      const bool up = (t & o) != 0;
#pragma unroll
      for (int k = 0; k < n; ++k) {
        const double other = __shfl_xor_sync(0xffffffffu, up ? js[k] : js[k + n], o);
        js[k] = (up ? js[k + n] : js[k]) + other;
      }
      first += up ? n : 0;
      left = n;
      o >>= 1;
    }
  }
  const int rest = (o << 1) - 1;  // lanes below this mask hold partial sums of one density
  for (; o > 0; o >>= 1) js[0] += __shfl_xor_sync(0xffffffffu, js[0], o);
  if (store && (rest <= 0 || (t & rest) == 0)) {
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (k < left && first + k < d.nd) atomicAdd(d.J + (first + k) * d.dstride + elem, w * js[k]);
  }
}

// (s s|C) DF-J launches digesting per integral (digest == 1), lanes over the
// kets of 32 / warpW tiles: gamma_P[C] += w D_ab (ss|P)_C per lane,
// and J_ab += w_J sum over the tile's kets and C of (ss|P)_C c_PC, reduced
// across the tile's lanes into one add.  The same sums as the tile kernel's
// digest.  kMulti: up to eight densities (digest == 4), the integrals formed
// once; gamma and J by FP64 atomics as in the tile kernel.
template <int LC, bool kMulti>
__global__ void __launch_bounds__(kSsThreads) eri3c_ss_dfj_kernel(const __grid_constant__ ClassDesc d) {
  constexpr int NC = (LC + 1) * (LC + 2) / 2, NS = 2 * LC + 1;
  __shared__ double sP[kSsThreads * odd_stride(NC)];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double* row = sP + threadIdx.x * odd_stride(NC);
  const int W = d.warpW, NP = 32 / W, g = lane / W, t = lane - g * W;
  const long long nwarps = (long long)gridDim.x * (kSsThreads / 32);
  for (long long w0 = (blockIdx.x * (long long)(kSsThreads / 32) + warp) * NP; w0 < d.nwtiles; w0 += nwarps * NP) {
    const int4 tt = w0 + g < d.nwtiles ? __ldg(d.wtiles + w0 + g) : int4{0, 0, 0, 0};
    const int4 sp = __ldg(d.subpairs + tt.x);
    const long long pair = sp.x;
    const int4 pao = __ldg(d.pair_ao + pair);
    const double wg = pao.z ? 1.0 : 2.0, wj = pao.z ? 0.5 : 1.0;
    const long long elem = (long long)pao.x * d.ldD + pao.y;
    const double Dab = !kMulti && d.gacc ? __ldg(d.D + elem) : 0.0;
    double jsum = 0.0;
    double js[8];
    if (kMulti)
#pragma unroll
      for (int k = 0; k < 8; ++k) js[k] = 0.0;
    const bool live = t < tt.z;
    double acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = 0.0;
    const long long q = tt.y + t;
    if (live) {
      ss_prims<LC>(d, pair, sp, q, acc);
#pragma unroll
      for (int c = 0; c < NC; ++c) row[c] = acc[c];
      const int ao = __ldg(d.aux_ao + q);
#pragma unroll
      for (int C = 0; C < NS; ++C) {
        double v = 0.0;
        for (int k = __ldg(d.kptr + C); k < __ldg(d.kptr + C + 1); ++k) {
          const int2 e = __ldg(d.kent + k);
          v = fma(__ldg(d.pal + e.y), row[e.x], v);
        }
        if (kMulti) {
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            if (k >= d.nd) break;
            if (d.gamma) atomicAdd(d.gamma + k * d.cstride + ao + C, wg * v * __ldg(d.D + k * d.dstride + elem));
            if (d.J) js[k] = fma(v, __ldg(d.cvec + k * d.cstride + ao + C), js[k]);
          }
          continue;
        }
        if (d.gacc) fix_add(d.gacc + kFixWords * (ao + C), wg * Dab * v);
        if (d.Jacc) jsum = fma(v, __ldg(d.cvec + ao + C), jsum);
      }
    }
    if (kMulti) {
      if (d.J) multi_j(d, js, W, t, tt.z > 0, wj, elem);
    } else if (d.Jacc) {
      for (int o = W >> 1; o > 0; o >>= 1) jsum += __shfl_xor_sync(0xffffffffu, jsum, o);
      if (t == 0 && tt.z) fix_add(d.Jacc + kFixWords * elem, wj * jsum);
    }
  }
}

// (p s|C) classes, lc <= 4: la = 1, lb = 0 in the A orientation, or the
// (s p|C) class run B-oriented (recurrences on the p shell, no HRR; its
// descriptor holds the (p s|C) tables with orient = 1).  With
// a = 1_i the n-quantum CVRR2 has two terms,
//   (1_i 0|c) = (1_i 0)_{0,c} + c_i (0 0)_{1,c-1_i}    (Eq. cVRR2),
// whose prerequisites are A_i(c) = sum [1_i 0|0]^(lc) X^c and
// B(n) = sum [00|0]^(lc) Y X^n (Eq. a0cv2, Y = 1/(2(gamma+zeta_c))), with
// [1_i 0|0]^(lc) = PA_i [00|0]^(lc) - (rho/gamma) PC_i [00|0]^(lc+1)
// (Eq. vrr1): 3 ncart(lc) + ncart(lc-1) accumulators held in registers.
constexpr int kPsThreads = 64;

template <int LC>
__device__ __forceinline__ void ps_prims(const ClassDesc& d, long long pair, const int4& sp, long long q,
                                         double (&A)[3][(LC + 1) * (LC + 2) / 2], double* Bm) {
  const double Cx = __ldg(d.auxc + 3 * q), Cy = __ldg(d.auxc + 3 * q + 1), Cz = __ldg(d.auxc + 3 * q + 2);
  const int fpa = d.orient ? PR_PB : PR_PA;
  for (int ip = 0; ip < sp.z; ++ip) {
    const double* pr = d.pairrec + (pair * d.Kab_rec + __ldg(d.primidx + sp.y + ip)) * kPairRec;
    const double gam = __ldg(pr + PR_G), K = __ldg(pr + PR_K);
    const double PAx = __ldg(pr + fpa), PAy = __ldg(pr + fpa + 1), PAz = __ldg(pr + fpa + 2);
    const double PCx = __ldg(pr + PR_P) - Cx, PCy = __ldg(pr + PR_P + 1) - Cy, PCz = __ldg(pr + PR_P + 2) - Cz;
    const double pc2 = fma(PCz, PCz, fma(PCy, PCy, PCx * PCx));
    for (int ic = 0; ic < d.Kc; ++ic) {
      const double zc = __ldg(d.auxrec + (q * d.Kc + ic) * kAuxRec);
      const double ccp = __ldg(d.auxrec + (q * d.Kc + ic) * kAuxRec + 1);
      const double sg = gam + zc;
      const double rs = rsqrt_fp64(sg);
      const double r = rs * rs;
      const double gr = gam * r, rg = zc * r;
      const double Tb = gr * zc * pc2;
      double v2[2];
      boys_scaled(d.boys_tab, d.boys_mid, d.boys_cL, LC + 1, LC, Tb, K * ccp * rs, v2, 1);
      const double V0 = v2[0];
      const double Vx = fma(-rg * PCx, v2[1], PAx * V0), Vy = fma(-rg * PCy, v2[1], PAy * V0),
                   Vz = fma(-rg * PCz, v2[1], PAz * V0);
      double px[LC + 1], py[LC + 1], pz[LC + 1];
      px[0] = 1.0; py[0] = 1.0; pz[0] = 1.0;
      const double Xx = gr * PCx, Xy = gr * PCy, Xz = gr * PCz;
#pragma unroll
      for (int j = 1; j <= LC; ++j) {
        px[j] = px[j - 1] * Xx;
        py[j] = py[j - 1] * Xy;
        pz[j] = pz[j - 1] * Xz;
      }
      int c = 0;
#pragma unroll
      for (int nx = LC; nx >= 0; --nx)
#pragma unroll
        for (int ny = LC - nx; ny >= 0; --ny) {
          const double m = px[nx] * (py[ny] * pz[LC - nx - ny]);
          A[0][c] = fma(Vx, m, A[0][c]);
          A[1][c] = fma(Vy, m, A[1][c]);
          A[2][c] = fma(Vz, m, A[2][c]);
          ++c;
        }
      if (LC > 0) {
        const double VY = V0 * (0.5 * r);
        int n = 0;
#pragma unroll
        for (int nx = LC - 1; nx >= 0; --nx)
#pragma unroll
          for (int ny = LC - 1 - nx; ny >= 0; --ny) {
            Bm[n] = fma(VY, px[nx] * (py[ny] * pz[LC - 1 - nx - ny]), Bm[n]);
            ++n;
          }
      }
    }
  }
}

// The (p s|c) targets G(i, c) = A_i(c) + c_i B(c - 1_i) into row[i * NC + c].
template <int LC>
__device__ __forceinline__ void ps_targets(const double (&A)[3][(LC + 1) * (LC + 2) / 2], const double* Bm,
                                           double* row) {
  constexpr int NC = (LC + 1) * (LC + 2) / 2;
  int c = 0;
#pragma unroll
  for (int nx = LC; nx >= 0; --nx)
#pragma unroll
    for (int ny = LC - nx; ny >= 0; --ny) {
      const int nz = LC - nx - ny;
      // index of c - 1_i in the Cartesian order of degree LC-1
      double gx = A[0][c], gy = A[1][c], gz = A[2][c];
      if (LC > 0) {
        // position of (x, y, z) of degree LC-1: (LC-1-x)(LC-x)/2 + (LC-1-x-y)
        if (nx > 0) gx = fma((double)nx, Bm[(LC - nx) * (LC - nx + 1) / 2 + (LC - nx - ny)], gx);
        if (ny > 0) gy = fma((double)ny, Bm[(LC - 1 - nx) * (LC - nx) / 2 + (LC - nx - ny)], gy);
        if (nz > 0) gz = fma((double)nz, Bm[(LC - 1 - nx) * (LC - nx) / 2 + (LC - 1 - nx - ny)], gz);
      }
      row[c] = gx;
      row[NC + c] = gy;
      row[2 * NC + c] = gz;
      ++c;
    }
}

// Ket then bra transform of one triple's targets (row: 3 x NC) into
// out[s * NS + C], s the bra component in storage order.
template <int LC>
__device__ __forceinline__ void ps_transform(const ClassDesc& d, const double* row, double* out) {
  constexpr int NC = (LC + 1) * (LC + 2) / 2, NS = 2 * LC + 1;
  double H[3][NS];
#pragma unroll
  for (int C = 0; C < NS; ++C) {
    double v0 = 0.0, v1 = 0.0, v2 = 0.0;
    for (int k = __ldg(d.kptr + C); k < __ldg(d.kptr + C + 1); ++k) {
      const int2 e = __ldg(d.kent + k);
      const double w = __ldg(d.pal + e.y);
      v0 = fma(w, row[e.x], v0);
      v1 = fma(w, row[NC + e.x], v1);
      v2 = fma(w, row[2 * NC + e.x], v2);
    }
    H[0][C] = v0;
    H[1][C] = v1;
    H[2][C] = v2;
  }
  if (d.nbA) {
#pragma unroll
    for (int A = 0; A < 3; ++A) {
      const int q0 = __ldg(d.baptr + A), q1 = __ldg(d.baptr + A + 1);
#pragma unroll
      for (int C = 0; C < NS; ++C) {
        double v = 0.0;
        for (int k = q0; k < q1; ++k) {
          const int2 e = __ldg(d.baent + k);
          // a single 3-way select keeps H in registers
          const double h = e.x == 0 ? H[0][C] : (e.x == 1 ? H[1][C] : H[2][C]);
          v = fma(__ldg(d.pal + e.y), h, v);
        }
        out[A * NS + C] = v;
      }
    }
  } else {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int C = 0; C < NS; ++C) out[a * NS + C] = H[a][C];
  }
}

template <int LC>
__global__ void __launch_bounds__(kPsThreads) eri3c_ps_kernel(const __grid_constant__ ClassDesc d) {
  constexpr int NC = (LC + 1) * (LC + 2) / 2, NS = 2 * LC + 1, NB = 3 * NS;
  constexpr int NCM = LC > 0 ? LC * (LC + 1) / 2 : 1;
  __shared__ double sG[kPsThreads * odd_stride(3 * NC)];
  __shared__ double sO[kPsThreads * NB];
  __shared__ long long sOff[kPsThreads];
  __shared__ int sAcc[kPsThreads];
  const int tid = threadIdx.x;
  const long long ntri = d.nsub * d.naux;
  for (long long base = (long long)blockIdx.x * kPsThreads; base < ntri; base += (long long)gridDim.x * kPsThreads) {
    const long long w = base + tid;
    long long off = -1;
    int accum = 0;
    if (w < ntri) {
      double A[3][NC], Bm[NCM];
#pragma unroll
      for (int c = 0; c < NC; ++c) A[0][c] = A[1][c] = A[2][c] = 0.0;
#pragma unroll
      for (int n = 0; n < NCM; ++n) Bm[n] = 0.0;
      const long long sub = w / d.naux;
      const long long q = w - sub * d.naux;
      const int4 sp = __ldg(d.subpairs + sub);
      accum = sp.w == 1;
      off = (((long long)sp.x - d.out_pair0) * d.naux + q) * (long long)d.nblk;
      ps_prims<LC>(d, sp.x, sp, q, A, Bm);
      double* row = sG + tid * odd_stride(3 * NC);
      ps_targets<LC>(A, Bm, row);
      ps_transform<LC>(d, row, sO + tid * NB);
    }
    sOff[tid] = off;
    sAcc[tid] = accum;
    __syncthreads();
    for (int i = tid; i < kPsThreads * NB; i += kPsThreads) {
      const int t = i / NB, x = i - t * NB;
      const long long o = sOff[t];
      if (o < 0) continue;
      double v = sO[i];
      if (sAcc[t]) v += d.out[o + x];
      d.out[o + x] = v;
    }
    __syncthreads();
  }
}

// (p s|C) DF-J launches digesting per integral, lanes over the kets of 32 /
// warpW tiles as in eri3c_ss_dfj_kernel: gamma_P[C] += w sum_s D_s (ps|P)_{sC}
// per lane and J_s += w_J sum over the tile's kets and C of (ps|P)_{sC} c_PC,
// reduced across the tile's lanes.  kMulti: up to eight densities.
template <int LC, bool kMulti>
__global__ void __launch_bounds__(kPsThreads) eri3c_ps_dfj_kernel(const __grid_constant__ ClassDesc d) {
  constexpr int NC = (LC + 1) * (LC + 2) / 2, NS = 2 * LC + 1, NB = 3 * NS;
  constexpr int NCM = LC > 0 ? LC * (LC + 1) / 2 : 1;
  __shared__ double sG[kPsThreads * odd_stride(3 * NC)];
  __shared__ double sO[kPsThreads * NB];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double* row = sG + threadIdx.x * odd_stride(3 * NC);
  double* out = sO + threadIdx.x * NB;
  const int W = d.warpW, NP = 32 / W, g = lane / W, t = lane - g * W;
  const long long nwarps = (long long)gridDim.x * (kPsThreads / 32);
  for (long long w0 = (blockIdx.x * (long long)(kPsThreads / 32) + warp) * NP; w0 < d.nwtiles; w0 += nwarps * NP) {
    const int4 tt = w0 + g < d.nwtiles ? __ldg(d.wtiles + w0 + g) : int4{0, 0, 0, 0};
    const int4 sp = __ldg(d.subpairs + tt.x);
    const long long pair = sp.x;
    const int4 pao = __ldg(d.pair_ao + pair);
    const double wg = pao.z ? 1.0 : 2.0, wj = pao.z ? 0.5 : 1.0;
    const long long elem = (long long)pao.x * d.ldD + pao.y, step = d.orient ? 1 : d.ldD;
    double Ds[3] = {0.0, 0.0, 0.0};
    if (!kMulti && d.gacc)
#pragma unroll
      for (int s = 0; s < 3; ++s) Ds[s] = __ldg(d.D + elem + s * step);
    double jm[3][8];
    if (kMulti)
#pragma unroll
      for (int k = 0; k < 24; ++k) jm[k >> 3][k & 7] = 0.0;
    double js[3] = {0.0, 0.0, 0.0};
    if (t < tt.z) {
      const long long q = tt.y + t;
      double A[3][NC], Bm[NCM];
#pragma unroll
      for (int c = 0; c < NC; ++c) A[0][c] = A[1][c] = A[2][c] = 0.0;
#pragma unroll
      for (int n = 0; n < NCM; ++n) Bm[n] = 0.0;
      ps_prims<LC>(d, pair, sp, q, A, Bm);
      ps_targets<LC>(A, Bm, row);
      ps_transform<LC>(d, row, out);
      const int ao = __ldg(d.aux_ao + q);
      if (kMulti) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          if (k >= d.nd) break;
          const double* D = d.D + k * d.dstride + elem;
          double D0 = 0.0, D1 = 0.0, D2 = 0.0;
          if (d.gamma) { D0 = __ldg(D); D1 = __ldg(D + step); D2 = __ldg(D + 2 * step); }
#pragma unroll
          for (int C = 0; C < NS; ++C) {
            const double i0 = out[C], i1 = out[NS + C], i2 = out[2 * NS + C];
            if (d.gamma) atomicAdd(d.gamma + k * d.cstride + ao + C, wg * fma(D0, i0, fma(D1, i1, D2 * i2)));
            if (d.J) {
              const double cv = __ldg(d.cvec + k * d.cstride + ao + C);
              jm[0][k] = fma(i0, cv, jm[0][k]);
              jm[1][k] = fma(i1, cv, jm[1][k]);
              jm[2][k] = fma(i2, cv, jm[2][k]);
            }
          }
        }
      } else
#pragma unroll
      for (int C = 0; C < NS; ++C) {
        const double i0 = out[C], i1 = out[NS + C], i2 = out[2 * NS + C];
        if (d.gacc) fix_add(d.gacc + kFixWords * (ao + C), wg * fma(Ds[0], i0, fma(Ds[1], i1, Ds[2] * i2)));
        if (d.Jacc) {
          const double cv = __ldg(d.cvec + ao + C);
          js[0] = fma(i0, cv, js[0]);
          js[1] = fma(i1, cv, js[1]);
          js[2] = fma(i2, cv, js[2]);
        }
      }
    }
    if (kMulti) {
      if (d.J)
#pragma unroll
        for (int s = 0; s < 3; ++s) multi_j(d, jm[s], W, t, tt.z > 0, wj, elem + s * step);
    } else if (d.Jacc) {
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        double v = js[s];
        for (int o = W >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (t == 0 && tt.z) {
          fix_add(d.Jacc + kFixWords * (elem + s * step), wj * v);
        }
      }
    }
  }
}

// Persistent form for mixed workloads: every CTA pulls (descriptor, tile)
// work items from one atomic counter until the list is exhausted (items are
// ordered longest first on the host).  No CTA ever waits on another.  The
// item's descriptor is staged in shared memory (re-copied only when the class
// changes), so the tile body reads its fields from there, not from global
// memory.  kMinBlocks = 2 caps the registers at 64 so that two 512-thread
// CTAs fit an SM, kMinBlocks = 1 (items whose shared memory lets only one fit)
// leaves the compiler free.
constexpr int kPersThreads = 512;

template <int kMinBlocks>
__global__ void __launch_bounds__(kPersThreads, kMinBlocks) eri3c_persistent(const ClassDesc* __restrict__ descs,
                                                                         const int2* __restrict__ work, long long nwork,
                                                                         unsigned long long* __restrict__ counter) {
  extern __shared__ double sm[];
  __shared__ __align__(16) ClassDesc sd;
  __shared__ long long next;
  int cur = -1;
  constexpr int kWords = (int)(sizeof(ClassDesc) / 8);
  static_assert(sizeof(ClassDesc) % 8 == 0, "descriptor copy in 8-byte words");
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) next = (long long)atomicAdd(counter, 1ULL);
    __syncthreads();
    const long long w = next;
    if (w >= nwork) return;
    const int2 wk = work[w];
    if (wk.x != cur) {
      const unsigned long long* src = reinterpret_cast<const unsigned long long*>(descs + wk.x);
      unsigned long long* dst = reinterpret_cast<unsigned long long*>(&sd);
      for (int i = threadIdx.x; i < kWords; i += kPersThreads) dst[i] = src[i];
      cur = wk.x;
      __syncthreads();
    }
    tile_body<0, kPersThreads>(sd, wk.y, sm);
  }
}

// Boys function evaluation for lx3c_boys: out[i*(mmax+1)+m] = F_m(T[i]).
__global__ void boys_kernel(const double* __restrict__ Tv, long long n, int mmax, const double* __restrict__ tab,
                            const double* __restrict__ mid, double cL, double* __restrict__ out) {
  long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  boys_scaled(tab, mid, cL, mmax, 0, Tv[i], 1.0, out + i * (mmax + 1), 1);
}

// ---------------------------------------------------------------------------
// host-side launch helpers (called from capi.cu)
// ---------------------------------------------------------------------------

// The current device's constants and the tile kernels' shared-memory limit (an
// attribute of the kernel on that device), with each device's first plan or
// allocation-free call.
cudaError_t init_constants() {
  double v[32];
  for (int m = 0; m < 32; ++m) v[m] = 1.0 / (2 * m + 1);
  cudaError_t e = cudaMemcpyToSymbol(c_inv2m1, v, sizeof(v));
  for (const void* f : {(const void*)eri3c_kernel<0, 512, 2>, (const void*)eri3c_kernel<0, 384, 3>,
                        (const void*)eri3c_kernel<1, 512, 2>, (const void*)eri3c_kernel<1, 384, 3>,
                        (const void*)eri3c_kernel_both})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
  return e;
}

cudaError_t launch_precompute(const DevBasis& orb, const int32_t* pairs, long long npair, int Ka, int Kb, double* rec,
                              double* ab, const DevBasis& aux, const int32_t* auxs, long long naux, int Kc,
                              double* auxrec, double* auxc, cudaStream_t st) {
  const long long n = npair * Ka * Kb + naux * Kc;
  if (n == 0) return cudaSuccess;
  precompute_kernel<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(orb, pairs, npair, Ka, Kb, rec, ab, aux, auxs, naux, Kc,
                                                                auxrec, auxc);
  return cudaGetLastError();
}

cudaError_t launch_precompute_jobs(const DevBasis& orb, const DevBasis& aux, const PrecomputeJob* jobs, int n,
                                   long long blocks, cudaStream_t st) {
  if (n == 0 || blocks == 0) return cudaSuccess;
  precompute_jobs_kernel<<<(unsigned)blocks, 128, 0, st>>>(orb, aux, jobs, n);
  return cudaGetLastError();
}

// SM count of the current device, for the grid-stride grids of the
// register-resident kernels (read once; 152 on GB300).
static int device_sms() {
  static const int n = [] {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0)
      v = 152;
    return v;
  }();
  return n;
}

// Whether three CTAs of the 384-thread tile kernel fit an SM.
static bool three_ctas(int smem_bytes) { return smem_bytes <= 233472 / 3 - 1024; }

// Whether a launch runs on a register-resident kernel: (s s|C), or (p s|C) and
// B-oriented (s p|C) (whose descriptor holds the (p s|C) tables with orient =
// 1) with 1 <= lc <= 4 or contracted; (p s|s) with one primitive per triple
// measured faster on the tile kernel.  Stores and per-integral DF-J, for one
// density or several, the latter with the kernels' own tiles (several densities
// on 16 atoms: these classes 9.3 of 26.3 ms on the tile kernel; the caller
// leaves out the tiles of launches too small for it).
static bool on_register_kernel(const ClassDesc& d) {
  if (d.digest != 0 && !((d.digest == 1 || d.digest == 4) && d.wtiles)) return false;
  if (d.la == 0 && d.lb == 0) return d.orient == 0;
  return d.la == 1 && d.lb == 0 && d.lc <= 4 && (d.lc > 0 || d.K > 1);
}
static bool on_tile_kernel(const ClassDesc& d) { return !on_register_kernel(d); }

template <int LC>
static void launch_ss(const ClassDesc& d, unsigned g, cudaStream_t st) {
  if (d.digest == 0) eri3c_ss_kernel<LC><<<g, kSsThreads, 0, st>>>(d);
  else if (d.digest == 1) eri3c_ss_dfj_kernel<LC, false><<<g, kSsThreads, 0, st>>>(d);
  else eri3c_ss_dfj_kernel<LC, true><<<g, kSsThreads, 0, st>>>(d);
}
template <int LC>
static void launch_ps(const ClassDesc& d, unsigned g, cudaStream_t st) {
  if (d.digest == 0) eri3c_ps_kernel<LC><<<g, kPsThreads, 0, st>>>(d);
  else if (d.digest == 1) eri3c_ps_dfj_kernel<LC, false><<<g, kPsThreads, 0, st>>>(d);
  else eri3c_ps_dfj_kernel<LC, true><<<g, kPsThreads, 0, st>>>(d);
}

bool can_launch_both(const ClassDesc& a, const ClassDesc& b) {
  return a.digest == 0 && b.digest == 0 && on_tile_kernel(a) && on_tile_kernel(b);
}

cudaError_t launch_eri3c_both(const ClassDesc& a, int ga, const ClassDesc& b, int gb, cudaStream_t st) {
  const int smem = std::max(a.smem_doubles, b.smem_doubles) * 8;
  eri3c_kernel_both<<<ga + gb, kBothThreads, smem, st>>>(a, b, ga);
  return cudaGetLastError();
}

cudaError_t launch_eri3c(const ClassDesc& d, int grid, cudaStream_t st) {
  if (on_register_kernel(d)) {
    const int threads = d.la ? kPsThreads : kSsThreads;
    const long long items = d.digest ? d.nwtiles : d.nsub * d.naux;
    const long long per = d.digest ? threads / d.warpW : threads;
    const unsigned g = (unsigned)std::min<long long>(std::max<long long>((items + per - 1) / per, 1),
                                                     (long long)device_sms() * (d.la ? 64 : 32));
    if (d.la == 0) {
      switch (d.lc) {
        case 0: launch_ss<0>(d, g, st); break;
        case 1: launch_ss<1>(d, g, st); break;
        case 2: launch_ss<2>(d, g, st); break;
        case 3: launch_ss<3>(d, g, st); break;
        case 4: launch_ss<4>(d, g, st); break;
        case 5: launch_ss<5>(d, g, st); break;
        default: launch_ss<6>(d, g, st); break;
      }
    } else {
      switch (d.lc) {
        case 0: launch_ps<0>(d, g, st); break;
        case 1: launch_ps<1>(d, g, st); break;
        case 2: launch_ps<2>(d, g, st); break;
        case 3: launch_ps<3>(d, g, st); break;
        default: launch_ps<4>(d, g, st); break;
      }
    }
  } else {
    const int smem = d.smem_doubles * 8;
    if (d.digest == 4) {
      if (three_ctas(smem)) eri3c_kernel<1, 384, 3><<<grid, 384, smem, st>>>(d);
      else eri3c_kernel<1, 512, 2><<<grid, 512, smem, st>>>(d);
    } else {
      if (three_ctas(smem)) eri3c_kernel<0, 384, 3><<<grid, 384, smem, st>>>(d);
      else eri3c_kernel<0, 512, 2><<<grid, 512, smem, st>>>(d);
    }
  }
  return cudaGetLastError();
}

cudaError_t launch_boys(const double* T, long long n, int mmax, const double* tab, const double* mid, double cL,
                        double* out, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  boys_kernel<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(T, n, mmax, tab, mid, cL, out);
  return cudaGetLastError();
}

// The dynamic shared-memory attribute is set by persistent_occupancy(), which
// callers run before any stream capture.
cudaError_t launch_persistent(const ClassDesc* descs, const int2* work, long long nwork, unsigned long long* counter,
                              int grid, int smem_bytes, int two, cudaStream_t st) {
  if (two)
    eri3c_persistent<2><<<grid, kPersThreads, smem_bytes, st>>>(descs, work, nwork, counter);
  else
    eri3c_persistent<1><<<grid, kPersThreads, smem_bytes, st>>>(descs, work, nwork, counter);
  return cudaGetLastError();
}

int persistent_occupancy(int smem_bytes, int two) {
  int nb = 0;
  const int cap = 232448 - (int)sizeof(ClassDesc) - 64;
  cudaError_t e;
  if (two) {
    cudaFuncSetAttribute(eri3c_persistent<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, eri3c_persistent<2>, kPersThreads, smem_bytes);
  } else {
    cudaFuncSetAttribute(eri3c_persistent<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, eri3c_persistent<1>, kPersThreads, smem_bytes);
  }
  if (e != cudaSuccess) return 1;
  return nb < 1 ? 1 : nb;
}

// CTAs of the tile kernel per SM: its launch bounds, or what the shared memory
// of an SM holds (233,472 bytes, 1 KB of it per CTA reserved).
int eri3c_occupancy(int smem_bytes) {
  return std::max(1, std::min(three_ctas(smem_bytes) ? 3 : 2, 233472 / (smem_bytes + 1024)));
}

}  // namespace lx3c
