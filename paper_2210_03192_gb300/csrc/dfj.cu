// Density-fitted Coulomb build (paper Sec. 3: a DF-J builder fed by an
// integral-digestion callable, so that integrals never reach global memory):
//   gamma_P = sum_{mu nu} (mu nu|P) D_{mu nu},   J_{mu nu} = sum_P (mu nu|P) c_P
// over all AO pairs (mu, nu) of a solid-harmonic orbital basis, evaluated on
// unique shell pairs a <= b (off-diagonal pairs weighted twice in gamma and
// mirrored into J).
//
// Setup (lx3c_dfj_plan): Schwarz-type screening estimates Q_ab, Q_P; every
// (la lb | lc) class group keeps its ket shells sorted by Q_P so that the
// ket shells surviving Q_ab Q_P >= tol for a pair form a prefix of the list.
// Execution: the (s s|C) and (p s|C) groups, and strongly contracted ones of low
// angular momentum, run the class kernels in digest mode on tabulated tiles
// (sub-pair, ket range); all others, and the gradient of every group, run in
// the Hermite basis (hermite.cu), which forms no integral.  gamma, J and the gradient are accumulated into
// exact fixed-point accumulators (fixed128.cuh), so the result does not
// depend on the order of the contributions; final kernels convert them to
// FP64 and symmetrise J.
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <fstream>
#include <sstream>
#include <map>
#include <memory>
#include <string>
#include <tuple>
#include <vector>

#include "../../include/lx3c.h"
#include "fixed128.cuh"
#include "hermite.h"
#include "lx3c_internal.h"
#include "primitives.h"

namespace lx3c {
cudaError_t launch_precompute(const DevBasis& orb, const int32_t* pairs, long long npair, int Ka, int Kb, double* rec,
                              double* ab, const DevBasis& aux, const int32_t* auxs, long long naux, int Kc,
                              double* auxrec, double* auxc, cudaStream_t st);
cudaError_t launch_eri3c(const ClassDesc& d, int grid, cudaStream_t st);
int eri3c_occupancy(int smem_bytes);
cudaError_t launch_persistent(const ClassDesc* descs, const int2* work, long long nwork, unsigned long long* counter,
                              int grid, int smem_bytes, int two, cudaStream_t st);
int persistent_occupancy(int smem_bytes, int two);
}  // namespace lx3c

using namespace lx3c;

namespace {

// Ket-count bound for the shape chooser from the tile fill: the largest T
// (a power of two up to 512, at least 2) at which this launch's tiles hold at
// least 80% screened triples, and never above the longest ket list.
long long fill_bound(const std::vector<int4>& sub, const std::vector<int>& counts, int cmax) {
  long long tot = 0;
  for (auto& s : sub) tot += counts[s.x];
  int pick = 1;
  for (int T = 512; T >= 1; T /= 2) {
    long long slots = 0;
    for (auto& s : sub) slots += (long long)((counts[s.x] + T - 1) / T) * T;
    if (tot * 5 >= slots * 4) { pick = T; break; }
  }
  return std::min<long long>(cmax, std::max(2, pick));
}


lx3c_status dfail(lx3c_status s, const std::string& m) {
  set_last_error("dfj: " + m);
  return s;
}

#define DCUDA(expr)                                                                                      \
  do {                                                                                                   \
    cudaError_t e_ = (expr);                                                                             \
    if (e_ != cudaSuccess) return dfail(LX3C_ECUDA, std::string(#expr) + ": " + cudaGetErrorString(e_)); \
  } while (0)

// J <- J + J^T (the digest accumulates each unique shell pair into one block;
// diagonal shell blocks carry half weight, so the sum is exact there too).
__global__ void symmetrize(double* J, long long n) {
  long long i = blockIdx.y * (long long)blockDim.y + threadIdx.y;
  long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n || j >= n || j < i) return;
  if (i == j) {
    J[i * n + i] *= 2.0;
  } else {
    const double s = J[i * n + j] + J[j * n + i];
    J[i * n + j] = s;
    J[j * n + i] = s;
  }
}

// out[i] = value of the fixed-point accumulator acc[i] (gamma, gradient)
__global__ void fix_finish(const unsigned long long* __restrict__ acc, long long n, double* __restrict__ out) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) out[i] = fix_decode(acc + kFixWords * i);
}

// J[i][j] = A[i][j] + A[j][i] from the accumulated unique-pair blocks A (the
// digest adds each unique shell pair's block once, diagonal shell blocks
// with half weight, so this is exact on the diagonal too)
__global__ void fix_finish_J(const unsigned long long* __restrict__ acc, long long n, double* __restrict__ J) {
  const long long i = blockIdx.y * (long long)blockDim.y + threadIdx.y;
  const long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n && j < n) J[i * n + j] = fix_decode(acc + kFixWords * (i * n + j)) + fix_decode(acc + kFixWords * (j * n + i));
}

cudaError_t launch_fix_finish(const unsigned long long* acc, long long n, double* out, cudaStream_t st) {
  fix_finish<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(acc, n, out);
  return cudaGetLastError();
}

cudaError_t launch_fix_finish_J(const unsigned long long* acc, long long n, double* J, cudaStream_t st) {
  dim3 blk(32, 8), grd((unsigned)((n + 31) / 32), (unsigned)((n + 7) / 8));
  fix_finish_J<<<grd, blk, 0, st>>>(acc, n, J);
  return cudaGetLastError();
}

// energy = sum_i c_i gamma_i (one block, fixed-order tree reduction)
__global__ void dot_energy(const double* __restrict__ c, const double* __restrict__ g, long long n, double* out) {
  __shared__ double part[256];
  double s = 0.0;
  for (long long i = threadIdx.x; i < n; i += 256) s = fma(c[i], g[i], s);
  part[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = part[0];
}

constexpr double kPi = 3.14159265358979323846;

// sqrt of a Schwarz-type estimate of max |(ab|ab)| for a shell pair: the
// (ss|ss) value of each primitive pair times the rms size of (x-A)^la (x-B)^lb
// under the product Gaussian.
double q_pair_raw(int la, int ka, const double* A, const double* ea, const double* ca, int lb, int kb,
                  const double* B, const double* eb, const double* cb) {
  double ab2 = 0;
  for (int x = 0; x < 3; ++x) ab2 += (A[x] - B[x]) * (A[x] - B[x]);
  double q = 0;
  for (int ia = 0; ia < ka; ++ia)
    for (int ib = 0; ib < kb; ++ib) {
      const double za = ea[ia], zb = eb[ib], g = za + zb;
      double pa2 = 0, pb2 = 0;
      for (int x = 0; x < 3; ++x) {
        const double P = (za * A[x] + zb * B[x]) / g;
        pa2 += (P - A[x]) * (P - A[x]);
        pb2 += (P - B[x]) * (P - B[x]);
      }
      q += std::fabs(ca[ia] * cb[ib]) * std::exp(-za * zb / g * ab2) *
           std::sqrt(2.0 * std::pow(kPi, 2.5) / (g * g * std::sqrt(2.0 * g))) * std::pow(pa2 + 0.5 / g, 0.5 * la) *
           std::pow(pb2 + 0.5 / g, 0.5 * lb);
    }
  return q;
}

double q_aux_raw(int l, int k, const double* e, const double* c) {
  double q = 0;
  for (int i = 0; i < k; ++i)
    q += std::fabs(c[i]) * std::sqrt(2.0 * std::pow(kPi, 2.5) / (e[i] * e[i] * std::sqrt(2.0 * e[i]))) *
         std::pow(0.5 / e[i], 0.5 * l);
  return q;
}

double q_pair(const lx3c_basis* b, int sa, int sb) {
  return q_pair_raw(b->l[sa], b->k[sa], &b->xyz[3 * sa], &b->exps[b->off[sa]], &b->coefs[b->off[sa]], b->l[sb],
                    b->k[sb], &b->xyz[3 * sb], &b->exps[b->off[sb]], &b->coefs[b->off[sb]]);
}

double q_aux(const lx3c_basis* b, int s) { return q_aux_raw(b->l[s], b->k[s], &b->exps[b->off[s]], &b->coefs[b->off[s]]); }

// The estimate Q_ab Q_P is not a bound: on jittered clusters of the DF-J
// recipe the largest element of a triple reaches ~11x it (compact same-shell
// pairs).  A triple is kept when kSchwarzSafety Q_ab Q_P >= tol, so that the
// dropped triples stay below tol with that margin.
constexpr double kSchwarzSafety = 20.0;

// Ket shells a pair keeps: the prefix of the list (sorted by decreasing Q_P)
// with kSchwarzSafety Q_ab Q_P >= tol.
int kets_kept(double qpair, const std::vector<double>& qket, double tol) {
  const double thr = qpair > 0 ? tol / (kSchwarzSafety * qpair) : 1e308;
  int lo = 0, hi = (int)qket.size();
  while (lo < hi) {
    const int mid = (lo + hi) / 2;
    if (qket[mid] >= thr) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Every group runs in the Hermite basis except those whose integrals cost less.
// The Hermite form pays its two contractions per primitive triple, where the
// digestion of integrals is a few FMAs per contracted one: the groups with a
// register-resident class kernel, (s s|C) and (p s|C) with lc <= 4 (contracted
// when lc = 0), and strongly contracted ones of low angular momentum.  For these
// the line is drawn on operation counts.  Over 197 classes (la, lb <= 4, lc <= 4,
// 4 to 100 primitive triples a triple) the time of the Hermite form over the
// tile kernel's, gamma and J together, is, to 13 %, the ratio of their counts
// (the contracted stages taken 1.5 times), times 0.8 beyond lc = 0; the tile
// kernel is taken where that makes it a fifth faster (three tenths with two
// shells above s, where it scatters more).  ms before and after:
// (d s|s) K = 36 5.5 and 3.0, (f s|d) 16.1 and 10.6, (p p|s) 4.3 and 2.6; left in
// the Hermite basis: (p p|s) K = 4 0.54 (tile kernel 0.66), (f f|s) K = 36 4.2
// (5.3).  One route for every output: gamma or J alone are bit for bit those of
// both, which costs gamma alone, 0.6 of the Hermite form, up to a quarter at the
// line and little for lc = 0 ((p p|s) K = 36 2.51 and 2.57).
// Fewer than 12 primitive triples gain little and fewer tiles than SMs lose: the
// tile kernel runs a tile's primitives in chunks one after another, a Hermite
// launch spreads them ((d s|s) and (f s|s), K = 6, of 18 atoms 14.34 ms in the
// Hermite basis, 14.64 on the tile kernel).
bool use_hermite(const HermBra& b, const HermKet& k) {
  if (b.la + b.lb == 0) return false;
  if (b.la + b.lb == 1) return k.lc > 4 || (k.lc == 0 && b.Ka * b.Kb * k.Kc == 1);
  const double n = b.nprim * k.Kc;
  if (n < 12 || b.q.size() * ((k.shells.size() + 31) / 32) < 152) return true;
  try {
    const ClassTables& ct = class_tables(b.la, b.lb, k.lc, 1);
    const double nint = (2.0 * b.la + 1) * (2 * b.lb + 1) * (2 * k.lc + 1);
    const double tile = ct.flops_prim * n + 1.5 * (ct.flops_contr + 4.0 * nint);
    return (k.lc == 0 ? 1.0 : 0.8) * n * herm_class_flops(b.la + b.lb, k.lc) < (b.lb ? 1.3 : 1.2) * tile;
  } catch (std::exception&) {
    return true;  // no tile kernel for the class
  }
}

// Contributing primitive pairs of a bra class's shell pairs, averaged over up
// to 64 of them.
double mean_prims(const lx3c_basis* orb, const HermBra& b) {
  if (b.Ka * b.Kb < 4) return b.Ka * b.Kb;
  const size_t np = b.q.size(), step = std::max<size_t>(1, np / 64);
  long long kept = 0, seen = 0;
  std::vector<double> q(b.Ka * b.Kb), K(b.Ka * b.Kb);
  for (size_t i = 0; i < np; i += step, ++seen) {
    const int sa = b.pairs[2 * i], sb = b.pairs[2 * i + 1];
    double ab2 = 0, qmax = 0;
    for (int x = 0; x < 3; ++x) {
      const double d = orb->xyz[3 * sa + x] - orb->xyz[3 * sb + x];
      ab2 += d * d;
    }
    for (int r = 0; r < b.Ka * b.Kb; ++r) {
      const long long ia = orb->off[sa] + r / b.Kb, ib = orb->off[sb] + r % b.Kb;
      q[r] = prim_bound(orb->exps[ia], orb->coefs[ia], orb->exps[ib], orb->coefs[ib], ab2, b.la, b.lb, &K[r]);
      qmax = std::max(qmax, q[r]);
    }
    for (int r = 0; r < b.Ka * b.Kb; ++r) kept += prim_kept(K[r], q[r], qmax);
  }
  return (double)kept / (double)std::max(1LL, seen);
}

// One device allocation for everything a plan keeps: arrays to upload
// (copied at once) and work buffers.  Pointers are set by commit().  (A plan
// has some 25 arrays per class group; one allocation and one copy for each was
// 8 of the 18 ms that planning 12 atoms with g functions took.)
struct PlanArena {
  std::vector<char> up;
  size_t work = 0;
  std::vector<std::pair<void**, size_t>> fix_up, fix_work;
  template <class T>
  void add(T** ptr, const T* v, size_t n) {
    const size_t off = (up.size() + 255) & ~size_t(255);
    up.resize(off + std::max<size_t>(n, 1) * sizeof(T));
    if (n) std::memcpy(up.data() + off, v, n * sizeof(T));
    fix_up.push_back({(void**)ptr, off});
  }
  template <class T>
  void take(T** ptr, size_t n) {
    fix_work.push_back({(void**)ptr, work});
    work += (std::max<size_t>(n, 1) * sizeof(T) + 255) & ~size_t(255);
  }
  cudaError_t commit(char** base, cudaStream_t st) {
    const size_t first = (up.size() + 255) & ~size_t(255);
    cudaError_t e = cudaMalloc(base, std::max<size_t>(first + work, 256));
    if (e == cudaSuccess && !up.empty()) e = cudaMemcpyAsync(*base, up.data(), up.size(), cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    for (auto& f : fix_up) *f.first = *base + f.second;
    for (auto& f : fix_work) *f.first = *base + first + f.second;
    return cudaStreamSynchronize(st);
  }
};

struct DfjLaunch {
  ClassDesc desc;
  int grid = 1;
  long long ntiles = 0;
  int4* d_sub = nullptr;
  int* d_prim = nullptr;
  int4* d_tiles = nullptr;
  int4* d_wtiles = nullptr;  // register-resident kernels (ClassDesc::wtiles)
  bool own_tiles = false;  // re-tiled: d_tiles is its own allocation
  std::vector<int4> sub;   // host copy of the sub-pair list (re-tiling)
  int kmax = 0;
};

struct DfjGroup {
  int la, lb, lc, Ka, Kb, Kc;
  std::vector<int32_t> pairs, auxs, counts;
  std::vector<int> at;  // position of each pair in its bra class
  long long ntasks = 0;
  double flops = 0, nint = 0;
  int32_t* d_pairs = nullptr;
  int32_t* d_auxs = nullptr;
  int4* d_pair_ao = nullptr;
  int* d_aux_ao = nullptr;
  double* d_pairrec = nullptr;
  double* d_pairab = nullptr;
  double* d_auxrec = nullptr;
  double* d_auxc = nullptr;
  DfjLaunch L[2];
  // the group runs in the Hermite basis; its class launches L serve the
  // several-density build alone
  bool herm = false;
};

}  // namespace

struct lx3c_dfj {
  const lx3c_basis* orb = nullptr;
  const lx3c_basis* aux = nullptr;
  long long nao = 0, naux_ao = 0;
  double tol = 0;
  int natom = 0;
  int nsm = 0;
  bool gradient = false;
  std::vector<DfjGroup> groups;
  // records of every group: the groups outside the Hermite basis first
  PrecomputeJob* d_jobs = nullptr;
  int njobs = 0, njobs_plain = 0;
  long long job_blocks = 0, job_blocks_plain = 0;
  char* arena = nullptr;            // every device array of the groups, and the accumulators
  HermPlan* hj = nullptr;           // gamma and J of the Hermite groups
  HermPlan* hg = nullptr;           // gradient of every group
  // exact fixed-point accumulators per element: gamma, J, gradient
  unsigned long long* d_gacc = nullptr;
  unsigned long long* d_Jacc = nullptr;
  unsigned long long* d_facc = nullptr;
};

namespace lx3c {
const lx3c_basis* dfj_orbital_basis(const lx3c_dfj* plan) { return plan->orb; }
}  // namespace lx3c

extern "C" {

void lx3c_dfj_destroy(lx3c_dfj* p) {
  if (!p) return;
  for (auto& g : p->groups)
    for (auto& L : g.L)
      if (L.own_tiles) cudaFree(L.d_tiles);
  cudaFree(p->arena);
  herm_destroy(p->hj);
  herm_destroy(p->hg);
  delete p;
}

lx3c_status lx3c_dfj_plan(lx3c_dfj** out, const lx3c_basis* orb, const lx3c_basis* aux, double schwarz_tol,
                          int flags, void* stream) {
  if (!out) return dfail(LX3C_EINVAL, "null output pointer");
  *out = nullptr;
  if (!orb || !aux) return dfail(LX3C_EINVAL, "null basis");
  if (orb->nshell <= 0 || aux->nshell <= 0) return dfail(LX3C_EINVAL, "empty basis");
  if (!(schwarz_tol >= 0.0)) return dfail(LX3C_EINVAL, "negative or NaN tolerance");
  const bool want_grad = (flags & 1) != 0;
  for (int64_t s = 0; s < orb->nshell; ++s)
    if (orb->l[s] > LX3C_LMAX_ORB - (want_grad ? 1 : 0))
      return dfail(LX3C_ENOTSUP, "orbital shell beyond the supported l");
  if (want_grad) {
    for (int64_t s = 0; s < orb->nshell; ++s)
      if (orb->atom[s] < 0) return dfail(LX3C_EINVAL, "gradient needs an atom index on every shell");
    for (int64_t s = 0; s < aux->nshell; ++s)
      if (aux->atom[s] < 0) return dfail(LX3C_EINVAL, "gradient needs an atom index on every shell");
  }
  DevState* ds;
  int rc = device_state_get(&ds);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  std::unique_ptr<lx3c_dfj, void (*)(lx3c_dfj*)> p(new lx3c_dfj, lx3c_dfj_destroy);
  PlanArena arena;
  p->orb = orb;
  p->aux = aux;
  p->tol = schwarz_tol;
  p->nsm = dev_nsm(ds);
  std::vector<int> ao(orb->nshell + 1, 0), aq(aux->nshell + 1, 0);
  for (int64_t s = 0; s < orb->nshell; ++s) ao[s + 1] = ao[s] + 2 * orb->l[s] + 1;
  for (int64_t s = 0; s < aux->nshell; ++s) aq[s + 1] = aq[s] + 2 * aux->l[s] + 1;
  p->nao = ao[orb->nshell];
  p->naux_ao = aq[aux->nshell];
  p->gradient = want_grad;
  for (int64_t s = 0; s < orb->nshell; ++s) p->natom = std::max(p->natom, orb->atom[s] + 1);
  for (int64_t s = 0; s < aux->nshell; ++s) p->natom = std::max(p->natom, aux->atom[s] + 1);
  // ket shells by (l, K), sorted by decreasing Q_P
  std::map<std::pair<int, int>, std::vector<std::pair<double, int>>> kets;
  for (int64_t s = 0; s < aux->nshell; ++s) kets[{aux->l[s], aux->k[s]}].push_back({q_aux(aux, (int)s), (int)s});
  for (auto& kv : kets)
    std::sort(kv.second.begin(), kv.second.end(), [](auto& x, auto& y) { return x.first > y.first || (x.first == y.first && x.second < y.second); });
  // unique shell pairs, canonical orientation (l, K) of the first >= second
  std::map<std::tuple<int, int, int, int>, std::vector<std::pair<int, int>>> bra;
  std::map<std::tuple<int, int, int, int>, std::vector<double>> braq;
  for (int a = 0; a < (int)orb->nshell; ++a)
    for (int b = a; b < (int)orb->nshell; ++b) {
      int s1 = a, s2 = b;
      if (std::make_pair(orb->l[s1], orb->k[s1]) < std::make_pair(orb->l[s2], orb->k[s2])) std::swap(s1, s2);
      auto key = std::make_tuple(orb->l[s1], orb->k[s1], orb->l[s2], orb->k[s2]);
      bra[key].push_back({s1, s2});
      braq[key].push_back(q_pair(orb, s1, s2));
    }
  std::vector<HermBra> hbra;
  std::vector<HermKet> hket;
  for (auto& bk : bra) {
    HermBra h{std::get<0>(bk.first), std::get<2>(bk.first), std::get<1>(bk.first), std::get<3>(bk.first), {}, {}, 0.0};
    for (auto& e : bk.second) {
      h.pairs.push_back(e.first);
      h.pairs.push_back(e.second);
    }
    h.q = braq[bk.first];
    h.nprim = mean_prims(orb, h);
    hbra.push_back(std::move(h));
  }
  for (auto& kk : kets) {
    HermKet h{kk.first.first, kk.first.second, {}, {}};
    for (auto& e : kk.second) {
      h.shells.push_back(e.second);
      h.q.push_back(e.first);
    }
    hket.push_back(std::move(h));
  }
  for (auto& hb : hbra) {
    for (auto& hk : hket) {
      DfjGroup g;
      g.la = hb.la; g.Ka = hb.Ka;
      g.lb = hb.lb; g.Kb = hb.Kb;
      g.lc = hk.lc; g.Kc = hk.Kc;
      g.herm = use_hermite(hb, hk);
      g.auxs = hk.shells;
      for (size_t i = 0; i < hb.q.size(); ++i) {
        const int lo = kets_kept(hb.q[i], hk.q, schwarz_tol);
        if (lo == 0) continue;
        g.pairs.push_back(hb.pairs[2 * i]);
        g.pairs.push_back(hb.pairs[2 * i + 1]);
        g.counts.push_back(lo);
        g.at.push_back((int)i);
        g.ntasks += lo;
      }
      if (g.counts.empty()) continue;
      p->groups.push_back(std::move(g));
    }
  }
  rc = herm_build(&p->hj, orb, aux, hbra, hket, use_hermite, kets_kept, schwarz_tol, false, p->nao, st);
  if (!rc && want_grad)
    rc = herm_build(&p->hg, orb, aux, hbra, hket, [](const HermBra&, const HermKet&) { return true; }, kets_kept,
                    schwarz_tol, true, p->nao, st);
  if (rc) return rc;
  // contributions to one element of the gradient's fixed-point accumulators
  if (p->hg && herm_max_adds(p->hg) >= kFixMaxAdds)
    return dfail(LX3C_ENOTSUP, "gradient: an atom's force accumulator would take 2^32 or more contributions");
  // per group: orientation split (once per bra class: its groups follow one
  // another), tiles, device lists
  struct { std::tuple<int, int, int, int> key{-1, 0, 0, 0}; std::vector<std::array<int, 4>> at; std::vector<int> prim[2]; } memo;
  for (auto& g : p->groups) {
    if (memo.key != std::make_tuple(g.la, g.Ka, g.lb, g.Kb)) {
      memo.key = std::make_tuple(g.la, g.Ka, g.lb, g.Kb);
      memo.at.assign(bra[memo.key].size(), {-1, 0, 0, 0});  // first and count of each orientation
      memo.prim[0].clear();
      memo.prim[1].clear();
    }
    const long long np = (long long)g.counts.size(), na = (long long)g.auxs.size();
    const int nbra = (2 * g.la + 1) * (2 * g.lb + 1), nket = 2 * g.lc + 1;
    g.nint = (double)nbra * nket * (double)g.ntasks;
    std::vector<int4> sub[2];
    std::vector<int> prim[2];
    int kmax[2] = {0, 0}, cmax = 0;
    for (long long i = 0; i < np; ++i) {
      int oa = (int)prim[0].size(), ob = (int)prim[1].size();
      auto& m = memo.at[g.at[i]];
      if (m[0] < 0) {
        m[0] = (int)memo.prim[0].size();
        m[2] = (int)memo.prim[1].size();
        split_orientation(orb, g.pairs[2 * i], g.pairs[2 * i + 1], g.la, g.lb, memo.prim[0], memo.prim[1]);
        m[1] = (int)memo.prim[0].size() - m[0];
        m[3] = (int)memo.prim[1].size() - m[2];
      }
      const int na_ = m[1], nb_ = m[3];
      prim[0].insert(prim[0].end(), memo.prim[0].begin() + m[0], memo.prim[0].begin() + m[0] + na_);
      prim[1].insert(prim[1].end(), memo.prim[1].begin() + m[2], memo.prim[1].begin() + m[2] + nb_);
      if (na_) sub[0].push_back(int4{(int)i, oa, na_, 0});
      if (nb_) sub[1].push_back(int4{(int)i, ob, nb_, 0});
      kmax[0] = std::max(kmax[0], na_);
      kmax[1] = std::max(kmax[1], nb_);
      cmax = std::max(cmax, g.counts[i]);
    }
    std::vector<int4> pao(np);
    std::vector<int> aao(na);
    for (long long i = 0; i < np; ++i)
      pao[i] = int4{ao[g.pairs[2 * i]], ao[g.pairs[2 * i + 1]], g.pairs[2 * i] == g.pairs[2 * i + 1] ? 1 : 0, 0};
    for (long long q = 0; q < na; ++q) aao[q] = aq[g.auxs[q]];
    const int Kab = g.Ka * g.Kb;
    arena.add(&g.d_pairs, g.pairs.data(), g.pairs.size());
    arena.add(&g.d_auxs, g.auxs.data(), g.auxs.size());
    arena.add(&g.d_pair_ao, pao.data(), pao.size());
    arena.add(&g.d_aux_ao, aao.data(), aao.size());
    arena.take(&g.d_pairrec, (size_t)np * Kab * kPairRec);
    arena.take(&g.d_pairab, (size_t)np * 3);
    arena.take(&g.d_auxrec, (size_t)na * g.Kc * kAuxRec);
    arena.take(&g.d_auxc, (size_t)na * 3);
    for (int o = 0; o < 2; ++o) {
      if (sub[o].empty()) continue;
      DfjLaunch& L = g.L[o];
      const ClassTables* ct;
      try {
        ct = &class_tables(o ? g.lb : g.la, o ? g.la : g.lb, g.lc, 1);
      } catch (std::exception& e) {
        return dfail(LX3C_ENOTSUP, e.what());
      }
      DevClass* dc;
      rc = device_class_get(ds, *ct, &dc);
      if (rc) return rc;
      ClassDesc& d = L.desc;
      if (fill_class_desc(d, *ct, *dc, ds, o, kmax[o], Kab, g.Kc, fill_bound(sub[o], g.counts, cmax)) < 0)
        return dfail(LX3C_ENOTSUP, "class does not fit in shared memory");
      {
        // executed flops: each sub-pair's primitive pairs through this
        // orientation's primitive stages, its contracted stages and the
        // digestion (4 flops per integral) once per kept ket shell; in the
        // Hermite basis a fixed count per primitive triple
        double tris = 0, primtris = 0;
        for (auto& sp : sub[o]) {
          tris += g.counts[sp.x];
          primtris += (double)g.counts[sp.x] * sp.z * g.Kc;
        }
        g.flops += g.herm ? primtris * herm_class_flops(g.la + g.lb, g.lc)
                          : primtris * ct->flops_prim + tris * (ct->flops_contr + 4.0 * nbra * nket);
      }
      std::vector<int4> tiles;
      for (size_t s = 0; s < sub[o].size(); ++s) {
        const int cnt = g.counts[sub[o][s].x];
        for (int a0 = 0; a0 < cnt; a0 += d.T) tiles.push_back(int4{(int)s, a0, std::min(d.T, cnt - a0), 0});
      }
      L.ntiles = (long long)tiles.size();
      L.sub = sub[o];
      L.kmax = kmax[o];
      arena.add(&L.d_sub, sub[o].data(), sub[o].size());
      arena.add(&L.d_prim, prim[o].data(), prim[o].size());
      arena.add(&L.d_tiles, tiles.data(), tiles.size());
      if (!g.herm && g.la + g.lb <= 1) {
        // tiles of the register-resident kernel: the width that leaves fewest
        // lanes idle at the ends of the ket lists (a small charge for the
        // sub-pairs of unequal contraction that then share a warp), the most
        // contracted sub-pairs first.  (One tile of the tile kernel's T per
        // warp left half the lanes idle from f on: (s s|h) of 16 atoms 256
        // instructions per primitive triple where (s s|g) took 108.)
        double best = 1e300;
        for (int W = 32; W >= 1; W /= 2) {
          double slots = 0;
          for (auto& sp : sub[o]) slots += (double)((g.counts[sp.x] + W - 1) / W * W) * sp.z;
          slots *= 1.0 + 0.03 * (32 / W - 1);
          if (slots < 0.999 * best) { best = slots; d.warpW = W; }
        }
        std::vector<int4> wt;
        for (size_t s = 0; s < sub[o].size(); ++s) {
          const int cnt = g.counts[sub[o][s].x];
          for (int a0 = 0; a0 < cnt; a0 += d.warpW)
            wt.push_back(int4{(int)s, a0, std::min(d.warpW, cnt - a0), sub[o][s].z});
        }
        std::stable_sort(wt.begin(), wt.end(), [](const int4& x, const int4& y) { return x.w > y.w; });
        d.nwtiles = (long long)wt.size();
        arena.add(&L.d_wtiles, wt.data(), wt.size());
      }
      d.npair = np;
      d.naux = na;
      d.nsub = (long long)sub[o].size();
      d.ntiles = L.ntiles;
      d.ntile_aux = 1;
      d.digest = 1;
      set_digest_scratch(d);
      if ((long long)d.smem_doubles * 8 > 232448) return dfail(LX3C_ENOTSUP, "digestion scratch does not fit");
      d.ldD = p->nao;
      const int occ = eri3c_occupancy(d.smem_doubles * 8);
      L.grid = (int)std::min<long long>(L.ntiles, (long long)dev_nsm(ds) * occ * 8);
    }
  }
  arena.take(&p->d_gacc, (size_t)p->naux_ao * kFixWords);
  arena.take(&p->d_Jacc, (size_t)p->nao * p->nao * kFixWords);
  if (want_grad) arena.take(&p->d_facc, (size_t)p->natom * 3 * kFixWords);
  arena.take(&p->d_jobs, p->groups.size());
  DCUDA(arena.commit(&p->arena, st));
  for (auto& g : p->groups)
    for (auto& L : g.L) {
      if (!L.ntiles) continue;
      ClassDesc& d = L.desc;
      d.tiles = L.d_tiles; d.wtiles = L.d_wtiles; d.subpairs = L.d_sub; d.primidx = L.d_prim;
      d.pairrec = g.d_pairrec; d.pairab = g.d_pairab; d.auxrec = g.d_auxrec; d.auxc = g.d_auxc;
      d.pair_ao = g.d_pair_ao; d.aux_ao = g.d_aux_ao;
    }
  std::vector<PrecomputeJob> jobs;
  for (int herm = 0; herm < 2; ++herm) {
    for (auto& g : p->groups)
      if ((int)g.herm == herm) {
        jobs.push_back(PrecomputeJob{g.d_pairs, (long long)g.counts.size(), g.Ka, g.Kb, g.d_pairrec, g.d_pairab,
                                     g.d_auxs, (long long)g.auxs.size(), g.Kc, g.d_auxrec, g.d_auxc, p->job_blocks});
        p->job_blocks += jobs.back().blocks();
      }
    if (!herm) {
      p->njobs_plain = (int)jobs.size();
      p->job_blocks_plain = p->job_blocks;
    }
  }
  p->njobs = (int)jobs.size();
  if (!jobs.empty())
    DCUDA(cudaMemcpyAsync(p->d_jobs, jobs.data(), jobs.size() * sizeof(PrecomputeJob), cudaMemcpyHostToDevice, st));
  DCUDA(cudaStreamSynchronize(st));
  *out = p.release();
  return LX3C_OK;
}

// The pair and ket records of a plan's groups (all, or those that do not run in
// the Hermite basis).
static cudaError_t group_records(const lx3c_dfj* p, bool all, cudaStream_t st) {
  return launch_precompute_jobs(p->orb->dev(), p->aux->dev(), p->d_jobs, all ? p->njobs : p->njobs_plain,
                                all ? p->job_blocks : p->job_blocks_plain, st);
}

lx3c_status lx3c_dfj_execute(lx3c_dfj* p, const double* D, const double* c, double* gamma, double* J, void* stream) {
  if (!p) return dfail(LX3C_EINVAL, "null plan");
  if (!D || !c || (!gamma && !J)) return dfail(LX3C_EINVAL, "null pointer");
  cudaStream_t st = (cudaStream_t)stream;
  if (gamma) DCUDA(cudaMemsetAsync(p->d_gacc, 0, p->naux_ao * kFixBytes, st));
  if (J) DCUDA(cudaMemsetAsync(p->d_Jacc, 0, p->nao * p->nao * kFixBytes, st));
  if (p->hj) DCUDA(herm_execute(p->hj, D, c, gamma ? p->d_gacc : nullptr, J ? p->d_Jacc : nullptr, st));
  DCUDA(group_records(p, false, st));
  for (auto& g : p->groups) {
    if (g.herm) continue;
    for (auto& L : g.L) {
      if (!L.ntiles) continue;
      ClassDesc d = L.desc;
      d.D = D;
      d.cvec = c;
      d.gacc = gamma ? p->d_gacc : nullptr;
      d.Jacc = J ? p->d_Jacc : nullptr;
      DCUDA(launch_eri3c(d, L.grid, st));
    }
  }
  if (gamma) DCUDA(launch_fix_finish(p->d_gacc, p->naux_ao, gamma, st));
  if (J) DCUDA(launch_fix_finish_J(p->d_Jacc, p->nao, J, st));
  return LX3C_OK;
}

lx3c_status lx3c_dfj_execute_multi(lx3c_dfj* p, int nd, const double* D, const double* c, double* gamma, double* J,
                                   void* stream) {
  if (!p) return dfail(LX3C_EINVAL, "null plan");
  if (nd < 1 || nd > 8) return dfail(LX3C_EINVAL, "execute_multi: nd must be in 1..8");
  if ((gamma && !D) || (J && !c) || (!gamma && !J)) return dfail(LX3C_EINVAL, "execute_multi: null pointer");
  cudaStream_t st = (cudaStream_t)stream;
  const long long dstride = p->nao * p->nao, cstride = p->naux_ao;
  // check every launch's scratch before launching anything
  std::vector<ClassDesc> descs;
  std::vector<int> grids;
  for (auto& g : p->groups)
    for (auto& L : g.L) {
      if (!L.ntiles) continue;
      ClassDesc d = L.desc;
      d.digest = 4;
      d.nd = nd;
      d.dstride = dstride;
      d.cstride = cstride;
      d.D = D;
      d.cvec = c;
      d.gamma = gamma;
      d.J = J;
      const long long kAB = ((long long)d.onA * d.onB + 3) & ~3LL, kR = ((long long)d.T * d.nC + 3) & ~3LL;
      d.dscr = place_epilogue_scratch(d, 8 * (kAB + kR));
      // the register-resident kernels from two warps per SM on: a warp runs its
      // tiles' primitives, components and densities one after another, 170 us
      // for (s s|h) whatever the number of warps, where the tile kernel spreads
      // a tile over its threads (2 atoms, eight densities: 3.45 ms a build with
      // the register kernels, 2.73 without; 4 atoms 3.13 and 2.52, 16 atoms
      // 21.7 and 25.2)
      if (d.wtiles && (d.nwtiles * d.warpW + 31) / 32 < 2LL * p->nsm) d.wtiles = nullptr;
      if ((long long)d.smem_doubles * 8 > 232448) return dfail(LX3C_ENOTSUP, "execute_multi: scratch does not fit");
      descs.push_back(d);
      grids.push_back(L.grid);
    }
  if (gamma) DCUDA(cudaMemsetAsync(gamma, 0, (size_t)nd * cstride * 8, st));
  if (J) DCUDA(cudaMemsetAsync(J, 0, (size_t)nd * dstride * 8, st));
  size_t li = 0;
  DCUDA(group_records(p, true, st));
  for (auto& g : p->groups) {
    for (auto& L : g.L) {
      if (!L.ntiles) continue;
      DCUDA(launch_eri3c(descs[li], grids[li], st));
      ++li;
    }
  }
  if (J) {
    dim3 blk(32, 8), grd((unsigned)((p->nao + 31) / 32), (unsigned)((p->nao + 7) / 8));
    for (int k = 0; k < nd; ++k) symmetrize<<<grd, blk, 0, st>>>(J + k * dstride, p->nao);
    DCUDA(cudaGetLastError());
  }
  return LX3C_OK;
}

lx3c_status lx3c_dfj_energy(lx3c_dfj* p, const double* D, const double* c, double* gamma, double* energy,
                            void* stream) {
  if (!energy || !gamma) return dfail(LX3C_EINVAL, "null pointer");
  lx3c_status rc = lx3c_dfj_execute(p, D, c, gamma, nullptr, stream);
  if (rc) return rc;
  dot_energy<<<1, 256, 0, (cudaStream_t)stream>>>(c, gamma, p->naux_ao, energy);
  DCUDA(cudaGetLastError());
  return LX3C_OK;
}

lx3c_status lx3c_dfj_grad(lx3c_dfj* p, const double* D, const double* c, double* grad, void* stream) {
  if (!p) return dfail(LX3C_EINVAL, "null plan");
  if (!p->gradient) return dfail(LX3C_EINVAL, "plan was built without gradient support (flags & 1)");
  if (!D || !c || !grad) return dfail(LX3C_EINVAL, "null pointer");
  cudaStream_t st = (cudaStream_t)stream;
  DCUDA(cudaMemsetAsync(p->d_facc, 0, (size_t)p->natom * 3 * kFixBytes, st));
  if (p->hg) DCUDA(herm_gradient(p->hg, D, c, p->d_facc, st));
  DCUDA(launch_fix_finish(p->d_facc, (long long)p->natom * 3, grad, st));
  return LX3C_OK;
}

lx3c_status lx3c_schwarz_pair(int la, int ka, const double* A, const double* ea, const double* ca, int lb, int kb,
                              const double* B, const double* eb, const double* cb, double* q) {
  if (!A || !ea || !ca || !B || !eb || !cb || !q || la < 0 || lb < 0 || ka < 1 || kb < 1)
    return dfail(LX3C_EINVAL, "schwarz_pair: bad argument");
  *q = kSchwarzSafety * q_pair_raw(la, ka, A, ea, ca, lb, kb, B, eb, cb);
  return LX3C_OK;
}

lx3c_status lx3c_schwarz_aux(int l, int k, const double* e, const double* c, double* q) {
  if (!e || !c || !q || l < 0 || k < 1) return dfail(LX3C_EINVAL, "schwarz_aux: bad argument");
  *q = q_aux_raw(l, k, e, c);
  return LX3C_OK;
}

lx3c_status lx3c_dfj_info(const lx3c_dfj* p, double* out, int n) {
  if (!p || (!out && n > 0)) return dfail(LX3C_EINVAL, "null pointer");
  double tasks = 0, nint = 0, flops = 0, launches = 2, slots = 0;
  const double gflops = p->hg ? herm_flops(p->hg) : 0, glaunches = p->gradient ? 1 + (p->hg ? herm_launches(p->hg) : 0) : 0;
  if (p->hj) launches += herm_launches(p->hj);
  for (auto& g : p->groups) {
    for (auto& L : g.L) slots += (double)L.ntiles * L.desc.T;
    tasks += (double)g.ntasks;
    nint += g.nint;
    flops += g.flops;
    if (!g.herm) launches += (g.L[0].ntiles > 0) + (g.L[1].ntiles > 0);
  }
  launches += p->njobs_plain > 0;
  const double v[] = {(double)p->groups.size(), tasks, nint, flops, launches, (double)p->nao, (double)p->naux_ao,
                      (double)p->natom, gflops, glaunches, slots, p->hg ? herm_max_adds(p->hg) : 0.0};
  for (int i = 0; i < n && i < 12; ++i) out[i] = v[i];
  return LX3C_OK;
}

lx3c_status lx3c_dfj_group(const lx3c_dfj* p, int gi, int32_t* info, int32_t* pairs, int32_t* counts,
                           int32_t* auxs) {
  if (!p) return dfail(LX3C_EINVAL, "null plan");
  if (gi < 0 || gi >= (int)p->groups.size()) return dfail(LX3C_EINVAL, "group index out of range");
  const DfjGroup& g = p->groups[gi];
  if (info) {
    const int32_t v[] = {g.la, g.lb, g.lc, g.Ka, g.Kb, g.Kc, (int32_t)g.counts.size(), (int32_t)g.auxs.size()};
    std::memcpy(info, v, sizeof(v));
  }
  if (pairs) std::memcpy(pairs, g.pairs.data(), g.pairs.size() * 4);
  if (counts) std::memcpy(counts, g.counts.data(), g.counts.size() * 4);
  if (auxs) std::memcpy(auxs, g.auxs.data(), g.auxs.size() * 4);
  return LX3C_OK;
}


}  // extern "C"

// ---------------------------------------------------------------------------
// Batched uneven workloads: several molecules' DF-J builds, every class mixed,
// as one persistent kernel captured in a CUDA graph (not in the paper).
// ---------------------------------------------------------------------------

namespace {

// Shape of one (class, orientation, kmax, Kc) launch: triples per tile T.
std::string shape_key(const ClassDesc& d) {
  char b[96];
  std::snprintf(b, sizeof(b), "%d,%d,%d,%d,%d,%d,%d", d.la, d.lb, d.lc, d.bra_pure, d.Kab, d.Kc, d.digest);
  return b;
}

// Re-tile one launch for triples-per-tile T (other shape fields recomputed by
// the planner for that T); returns false if T does not fit.
bool retile(DfjLaunch& L, const DfjGroup& g, const DevState* ds, int T) {
  const ClassTables& ct = class_tables(L.desc.la, L.desc.lb, L.desc.lc, L.desc.bra_pure);
  ClassDesc d = L.desc;
  const int mode = T >= 32 ? 0 : 1;
  // keep G from the planner's choice for this T
  LaunchShape sh = largest_tile(ct, L.kmax, d.Kc, T, dev_smem(ds), 2);
  sh.T = T;
  sh.mode = mode;
  ClassDesc nd = d;
  fill_layout(nd, ct, sh);
  set_digest_scratch(nd);
  if ((long long)nd.smem_doubles * 8 > 232448 - 64) return false;
  nd.nchunk = (nd.K + nd.G - 1) / nd.G;
  std::vector<int4> tiles;
  for (size_t s2 = 0; s2 < L.sub.size(); ++s2) {
    const int cnt = g.counts[L.sub[s2].x];
    for (int a0 = 0; a0 < cnt; a0 += T) tiles.push_back(int4{(int)s2, a0, std::min(T, cnt - a0), 0});
  }
  int4* dt = nullptr;
  if (cudaMalloc(&dt, tiles.size() * sizeof(int4)) != cudaSuccess) return false;
  cudaMemcpy(dt, tiles.data(), tiles.size() * sizeof(int4), cudaMemcpyHostToDevice);
  if (L.own_tiles) cudaFree(L.d_tiles);
  L.d_tiles = dt;
  L.own_tiles = true;
  L.ntiles = (long long)tiles.size();
  nd.tiles = dt;
  nd.ntiles = L.ntiles;
  L.desc = nd;
  const int occ = eri3c_occupancy(nd.smem_doubles * 8);
  L.grid = (int)std::min<long long>(L.ntiles, (long long)dev_nsm(ds) * occ * 8);
  return true;
}

}  // namespace

struct lx3c_batch {
  std::vector<lx3c_dfj*> mols;
  DevState* ds = nullptr;
  std::map<std::string, int> tuned;   // shape_key -> T
  int ntuned_measured = 0;
  // bound state
  ClassDesc* d_descs = nullptr;
  int2* d_work = nullptr;
  unsigned long long* d_counter = nullptr;  // one per tier
  long long nwork = 0;
  int ndesc = 0;
  int smem = 0;
  int grid = 0;
  // mode 1 splits the work items into occupancy tiers, each run by a
  // persistent kernel sized for the tier's largest item: items that fit two
  // CTAs per SM, then the rest
  struct Tier {
    long long off = 0, n = 0;
    int smem = 0, grid = 0, two = 0;
  };
  std::vector<Tier> tiers;
  cudaGraph_t graph = nullptr;        // mode 1: persistent kernels, one per tier
  cudaGraphExec_t exec = nullptr;
  cudaGraph_t graph2 = nullptr;       // mode 2: class launches on parallel branches
  cudaGraphExec_t exec2 = nullptr;
  long long branch_kernels = 0;
  std::vector<const double*> D, c;
  std::vector<double*> gamma, J;
  long long plain_launches = 0, graph_kernels = 0;
};

namespace {

constexpr int kBranches = 4;

// Mode 2: the same build as a graph whose class launches (the one-class kernel,
// descriptor in the parameter space) are spread over kBranches parallel
// branches, longest first onto the least loaded branch; zeroing and
// precomputes come before the fork, J symmetrisation after the join.
cudaError_t capture_branches(lx3c_batch* b, const std::vector<ClassDesc>& descs, const std::vector<int>& grids,
                             const std::vector<std::pair<double, int>>& order, cudaStream_t cap) {
  if (b->exec2) { cudaGraphExecDestroy(b->exec2); b->exec2 = nullptr; }
  if (b->graph2) { cudaGraphDestroy(b->graph2); b->graph2 = nullptr; }
  cudaStream_t br[kBranches] = {};
  cudaEvent_t fork = nullptr, join[kBranches] = {};
  cudaError_t ce = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
  for (int i = 0; i < kBranches && ce == cudaSuccess; ++i) {
    ce = cudaStreamCreateWithFlags(&br[i], cudaStreamNonBlocking);
    if (ce == cudaSuccess) ce = cudaEventCreateWithFlags(&join[i], cudaEventDisableTiming);
  }
  if (ce == cudaSuccess) ce = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
  if (ce == cudaSuccess) {
    long long kernels = 0;
    const int nmol = (int)b->mols.size();
    for (int m = 0; m < nmol; ++m) {
      lx3c_dfj* p = b->mols[m];
      cudaMemsetAsync(p->d_gacc, 0, p->naux_ao * kFixBytes, cap);
      cudaMemsetAsync(p->d_Jacc, 0, p->nao * p->nao * kFixBytes, cap);
      group_records(p, false, cap);
      kernels += p->njobs_plain > 0;
    }
    cudaEventRecord(fork, cap);
    double load[kBranches] = {};
    for (int i = 0; i < kBranches; ++i) cudaStreamWaitEvent(br[i], fork, 0);
    // each molecule's Hermite chain on one branch, the largest first
    std::vector<int> by(nmol);
    for (int m = 0; m < nmol; ++m) by[m] = m;
    std::stable_sort(by.begin(), by.end(), [&](int x, int y) {
      return (b->mols[x]->hj ? herm_flops(b->mols[x]->hj) : 0) > (b->mols[y]->hj ? herm_flops(b->mols[y]->hj) : 0);
    });
    for (int m : by) {
      lx3c_dfj* p = b->mols[m];
      if (!p->hj) continue;
      int k = 0;
      for (int i = 1; i < kBranches; ++i)
        if (load[i] < load[k]) k = i;
      load[k] += herm_flops(p->hj);
      herm_execute(p->hj, b->D[m], b->c[m], p->d_gacc, p->d_Jacc, br[k]);
      kernels += herm_launches(p->hj);
    }
    for (auto& o : order) {
      int k = 0;
      for (int i = 1; i < kBranches; ++i)
        if (load[i] < load[k]) k = i;
      load[k] += o.first;
      launch_eri3c(descs[o.second], grids[o.second], br[k]);
      ++kernels;
    }
    for (int i = 0; i < kBranches; ++i) {
      cudaEventRecord(join[i], br[i]);
      cudaStreamWaitEvent(cap, join[i], 0);
    }
    for (int m = 0; m < nmol; ++m) {
      launch_fix_finish(b->mols[m]->d_gacc, b->mols[m]->naux_ao, b->gamma[m], cap);
      launch_fix_finish_J(b->mols[m]->d_Jacc, b->mols[m]->nao, b->J[m], cap);
      kernels += 2;
    }
    ce = cudaStreamEndCapture(cap, &b->graph2);
    if (ce == cudaSuccess) ce = cudaGraphInstantiate(&b->exec2, b->graph2, 0);
    b->branch_kernels = kernels;
  }
  for (int i = 0; i < kBranches; ++i) {
    if (br[i]) cudaStreamDestroy(br[i]);
    if (join[i]) cudaEventDestroy(join[i]);
  }
  if (fork) cudaEventDestroy(fork);
  return ce;
}

}  // namespace

extern "C" {

void lx3c_batch_destroy(lx3c_batch* b) {
  if (!b) return;
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  if (b->exec2) cudaGraphExecDestroy(b->exec2);
  if (b->graph2) cudaGraphDestroy(b->graph2);
  cudaFree(b->d_descs);
  cudaFree(b->d_work);
  cudaFree(b->d_counter);
  for (auto* m : b->mols) lx3c_dfj_destroy(m);
  delete b;
}

lx3c_status lx3c_batch_plan(lx3c_batch** out, int nmol, const lx3c_basis* const* orbs, const lx3c_basis* const* auxs,
                            double schwarz_tol, const char* tune_cache, void* stream) {
  if (!out) return dfail(LX3C_EINVAL, "null output pointer");
  *out = nullptr;
  if (nmol <= 0 || !orbs || !auxs) return dfail(LX3C_EINVAL, "empty molecule list");
  std::unique_ptr<lx3c_batch> b(new lx3c_batch);
  int rc = device_state_get(&b->ds);
  if (rc) return rc;
  for (int m = 0; m < nmol; ++m) {
    lx3c_dfj* p = nullptr;
    rc = lx3c_dfj_plan(&p, orbs[m], auxs[m], schwarz_tol, 0, stream);
    if (rc) return rc;
    b->mols.push_back(p);
  }
  // ---- autotuner: triples per tile for each launch signature, timed on the
  // signature's largest launch; results cached as "key T" lines.
  std::map<std::string, int> cache;
  if (tune_cache && *tune_cache) {
    std::ifstream f(tune_cache);
    std::string k;
    int T;
    while (f >> k >> T) cache[k] = T;
  }
  std::map<std::string, std::pair<DfjLaunch*, DfjGroup*>> biggest;
  for (auto* p : b->mols)
    for (auto& g : p->groups)
      for (auto& L : g.L) {
        if (!L.ntiles || g.herm) continue;
        const std::string k = shape_key(L.desc);
        auto it = biggest.find(k);
        long long work = (long long)L.desc.T * L.ntiles;
        if (it == biggest.end() || (long long)it->second.first->desc.T * it->second.first->ntiles < work)
          biggest[k] = {&L, &g};
      }
  cudaStream_t st = (cudaStream_t)stream;
  double *tg = nullptr, *tJ = nullptr, *tD = nullptr, *tc = nullptr;
  bool measured = false;
  for (auto& kv : biggest) {
    if (cache.count(kv.first)) {
      b->tuned[kv.first] = cache[kv.first];
      continue;
    }
    DfjLaunch& L = *kv.second.first;
    DfjGroup& g = *kv.second.second;
    lx3c_dfj* owner = nullptr;
    for (auto* p : b->mols)
      for (auto& gg : p->groups)
        if (&gg == &g) owner = p;
    if (!tg) {
      long long mx = 0, mxa = 0;
      for (auto* p : b->mols) { mx = std::max(mx, p->nao); mxa = std::max(mxa, p->naux_ao); }
      DCUDA(cudaMalloc(&tg, mxa * kFixBytes)); DCUDA(cudaMalloc(&tc, mxa * 8));
      DCUDA(cudaMalloc(&tJ, mx * mx * kFixBytes)); DCUDA(cudaMalloc(&tD, mx * mx * 8));
      DCUDA(cudaMemset(tg, 0, mxa * kFixBytes)); DCUDA(cudaMemset(tJ, 0, mx * mx * kFixBytes));
      DCUDA(cudaMemset(tc, 0, mxa * 8)); DCUDA(cudaMemset(tD, 0, mx * mx * 8));
    }
    DCUDA(launch_precompute(owner->orb->dev(), g.d_pairs, (long long)g.counts.size(), g.Ka, g.Kb, g.d_pairrec, g.d_pairab,
                            owner->aux->dev(), g.d_auxs, (long long)g.auxs.size(), g.Kc, g.d_auxrec, g.d_auxc, st));
    const int T0 = L.desc.T;
    std::vector<int> cands = {T0};
    if (T0 >= 2) cands.push_back(T0 / 2);
    if (T0 <= 256) cands.push_back(T0 * 2);
    float best = 1e30f;
    int bestT = T0;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    // time every candidate on the same prefix of sub-pairs: about 8 waves of
    // the planner's tiles, the same triples whatever T is
    long long nsub_t = (long long)L.sub.size();
    {
      const long long cap = 8LL * dev_nsm(b->ds) * 2;
      long long nt = 0;
      for (long long s2 = 0; s2 < (long long)L.sub.size(); ++s2) {
        nt += (g.counts[L.sub[s2].x] + T0 - 1) / T0;
        if (nt >= cap) { nsub_t = s2 + 1; break; }
      }
    }
    for (int T : cands) {
      if (!retile(L, g, b->ds, T)) continue;
      ClassDesc d = L.desc;
      d.wtiles = nullptr;  // the tile kernel, whose T this is
      d.D = tD; d.cvec = tc;
      d.gacc = (unsigned long long*)tg; d.Jacc = (unsigned long long*)tJ;
      long long nt = 0;
      for (long long s2 = 0; s2 < nsub_t; ++s2) nt += (g.counts[L.sub[s2].x] + T - 1) / T;
      d.ntiles = nt;
      const int grid = (int)std::min<long long>(nt, L.grid);
      launch_eri3c(d, grid, st);
      cudaEventRecord(e0, st);
      launch_eri3c(d, grid, st);
      cudaEventRecord(e1, st);
      cudaEventSynchronize(e1);
      float ms = 0;
      cudaEventElapsedTime(&ms, e0, e1);
      if (ms < best) { best = ms; bestT = T; }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    b->tuned[kv.first] = bestT;
    cache[kv.first] = bestT;
    measured = true;
    ++b->ntuned_measured;
  }
  cudaFree(tg); cudaFree(tJ); cudaFree(tD); cudaFree(tc);
  // apply the tuned shapes to every launch
  for (auto* p : b->mols)
    for (auto& g : p->groups)
      for (auto& L : g.L) {
        if (!L.ntiles || g.herm) continue;
        auto it = b->tuned.find(shape_key(L.desc));
        if (it != b->tuned.end() && it->second != L.desc.T) retile(L, g, b->ds, it->second);
      }
  if (measured && tune_cache && *tune_cache) {
    std::ofstream f(tune_cache);
    for (auto& kv : cache) f << kv.first << " " << kv.second << "\n";
  }
  DCUDA(cudaGetLastError());
  DCUDA(cudaStreamSynchronize(st));
  *out = b.release();
  return LX3C_OK;
}

lx3c_status lx3c_batch_bind(lx3c_batch* b, const double* const* D, const double* const* c, double* const* gamma,
                            double* const* J, void* stream) {
  if (!b || !D || !c || !gamma || !J) return dfail(LX3C_EINVAL, "null pointer");
  const int nmol = (int)b->mols.size();
  b->D.assign(D, D + nmol); b->c.assign(c, c + nmol);
  b->gamma.assign(gamma, gamma + nmol); b->J.assign(J, J + nmol);
  // descriptors with this binding's pointers, and the longest-first work list
  std::vector<ClassDesc> descs;
  std::vector<int> grids;
  std::vector<std::pair<double, int>> order;
  int smem = 0;
  b->plain_launches = 0;
  for (int m = 0; m < nmol; ++m) {
    lx3c_dfj* p = b->mols[m];
    b->plain_launches += 2 + (p->njobs_plain > 0) + (p->hj ? herm_launches(p->hj) : 0);
    for (auto& g : p->groups) {
      if (g.herm) continue;
      for (auto& L : g.L) {
        if (!L.ntiles) continue;
        ++b->plain_launches;
        ClassDesc d = L.desc;
        d.D = D[m]; d.cvec = c[m]; d.gacc = p->d_gacc; d.Jacc = p->d_Jacc;
        double fl = 0;
        lx3c_class_flops(d.la, d.lb, d.lc, d.Kab, d.Kc, 1, &fl);
        order.push_back({fl * (double)d.T * (double)L.ntiles, (int)descs.size()});
        descs.push_back(d);
        grids.push_back(L.grid);
        smem = std::max(smem, d.smem_doubles * 8);
      }
    }
  }
  std::stable_sort(order.begin(), order.end(), [](auto& x, auto& y) { return x.first > y.first; });
  // tiers: the items whose shared memory lets two CTAs fit an SM, then the
  // others; longest first within each tier
  std::vector<int2> work;
  b->tiers.clear();
  auto tier_of = [&](int sm) { return persistent_occupancy(sm, 1) >= 2 ? 0 : 1; };
  for (int tier = 0; tier < 2; ++tier) {
    lx3c_batch::Tier T;
    T.off = (long long)work.size();
    T.two = tier == 0 ? 1 : 0;
    for (auto& o : order) {
      const int sm = descs[o.second].smem_doubles * 8;
      if (tier_of(sm) != tier) continue;
      T.smem = std::max(T.smem, sm);
      for (long long t = 0; t < descs[o.second].ntiles; ++t) work.push_back(int2{o.second, (int)t});
    }
    T.n = (long long)work.size() - T.off;
    if (!T.n) continue;
    T.grid = dev_nsm(b->ds) * persistent_occupancy(T.smem, T.two);
    b->tiers.push_back(T);
  }
  cudaFree(b->d_descs);
  cudaFree(b->d_work);
  if (!b->d_counter) DCUDA(cudaMalloc(&b->d_counter, 3 * sizeof(unsigned long long)));
  DCUDA(cudaMalloc(&b->d_descs, descs.size() * sizeof(ClassDesc)));
  DCUDA(cudaMalloc(&b->d_work, std::max<size_t>(work.size(), 1) * sizeof(int2)));
  DCUDA(cudaMemcpy(b->d_descs, descs.data(), descs.size() * sizeof(ClassDesc), cudaMemcpyHostToDevice));
  DCUDA(cudaMemcpy(b->d_work, work.data(), work.size() * sizeof(int2), cudaMemcpyHostToDevice));
  b->nwork = (long long)work.size();
  b->ndesc = (int)descs.size();
  b->smem = smem;
  b->grid = b->tiers.empty() ? 0 : b->tiers[0].grid;
  // capture the whole batched build in one graph
  if (b->exec) { cudaGraphExecDestroy(b->exec); b->exec = nullptr; }
  if (b->graph) { cudaGraphDestroy(b->graph); b->graph = nullptr; }
  cudaStream_t cap;
  DCUDA(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
  DCUDA(cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal));
  b->graph_kernels = 0;
  for (int m = 0; m < nmol; ++m) {
    lx3c_dfj* p = b->mols[m];
    cudaMemsetAsync(p->d_gacc, 0, p->naux_ao * kFixBytes, cap);
    cudaMemsetAsync(p->d_Jacc, 0, p->nao * p->nao * kFixBytes, cap);
    group_records(p, false, cap);
    b->graph_kernels += p->njobs_plain > 0;
  }
  for (int m = 0; m < nmol; ++m) {
    lx3c_dfj* p = b->mols[m];
    if (!p->hj) continue;
    herm_execute(p->hj, D[m], c[m], p->d_gacc, p->d_Jacc, cap);
    b->graph_kernels += herm_launches(p->hj);
  }
  for (size_t t = 0; t < b->tiers.size(); ++t) {
    const auto& T = b->tiers[t];
    cudaMemsetAsync(b->d_counter + t, 0, sizeof(unsigned long long), cap);
    launch_persistent(b->d_descs, b->d_work + T.off, T.n, b->d_counter + t, T.grid, T.smem, T.two, cap);
    b->graph_kernels += 1;
  }
  for (int m = 0; m < nmol; ++m) {
    launch_fix_finish(b->mols[m]->d_gacc, b->mols[m]->naux_ao, gamma[m], cap);
    launch_fix_finish_J(b->mols[m]->d_Jacc, b->mols[m]->nao, J[m], cap);
    b->graph_kernels += 2;
  }
  cudaError_t ce = cudaStreamEndCapture(cap, &b->graph);
  if (ce != cudaSuccess) {
    cudaStreamDestroy(cap);
    return dfail(LX3C_ECUDA, std::string("graph capture: ") + cudaGetErrorString(ce));
  }
  ce = cudaGraphInstantiate(&b->exec, b->graph, 0);
  if (ce == cudaSuccess) ce = capture_branches(b, descs, grids, order, cap);
  cudaStreamDestroy(cap);
  if (ce != cudaSuccess) return dfail(LX3C_ECUDA, std::string("graph capture: ") + cudaGetErrorString(ce));
  (void)stream;
  return LX3C_OK;
}

lx3c_status lx3c_batch_execute(lx3c_batch* b, int mode, void* stream) {
  if (!b) return dfail(LX3C_EINVAL, "null batch");
  if (b->D.empty()) return dfail(LX3C_EINVAL, "batch not bound (lx3c_batch_bind)");
  cudaStream_t st = (cudaStream_t)stream;
  if (mode == 1 || mode == 2) {
    DCUDA(cudaGraphLaunch(mode == 1 ? b->exec : b->exec2, st));
    return LX3C_OK;
  }
  if (mode != 0) return dfail(LX3C_EINVAL, "mode must be 0, 1 or 2");
  for (size_t m = 0; m < b->mols.size(); ++m) {
    lx3c_status rc = lx3c_dfj_execute(b->mols[m], b->D[m], b->c[m], b->gamma[m], b->J[m], stream);
    if (rc) return rc;
  }
  return LX3C_OK;
}

lx3c_status lx3c_batch_info(const lx3c_batch* b, double* out, int n) {
  if (!b || (!out && n > 0)) return dfail(LX3C_EINVAL, "null pointer");
  double tasks = 0, nint = 0, flops = 0, slots = 0;
  for (auto* p : b->mols)
    for (auto& g : p->groups) {
      tasks += (double)g.ntasks; nint += g.nint; flops += g.flops;
      for (auto& L : g.L) slots += (double)L.ntiles * L.desc.T;
    }
  const double v[] = {(double)b->mols.size(), tasks, nint, flops, (double)b->plain_launches,
                      (double)b->graph_kernels, (double)b->nwork, (double)b->ndesc, (double)b->smem,
                      (double)b->grid, (double)b->tuned.size(), (double)b->ntuned_measured,
                      (double)b->branch_kernels, (double)kBranches, slots, (double)b->tiers.size()};
  for (int i = 0; i < n && i < 16; ++i) out[i] = v[i];
  return LX3C_OK;
}

}  // extern "C"
