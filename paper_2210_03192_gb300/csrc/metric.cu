// Density-fitting metric and solve (the step between gamma and J in a DF-J
// build, Sec. 1 and Sec. 4 of arXiv:2210.03192: the fitted density is
// c = V^{-1} gamma with V_PQ = (P|Q) over the auxiliary basis):
//   lx3c_metric_plan/execute  V_PQ = (P|Q) by the class kernel, as the
//                              3-centre integral (P 1|Q) whose bra partner is
//                              the constant function 1 (an s Gaussian with
//                              exponent 0), stored straight into V
//   lx3c_cholesky             blocked right-looking Cholesky V = L L^T in FP64
//   lx3c_cholesky_solve       L L^T X = B by blocked forward and backward
//                              substitution
//   lx3c_dfj_coulomb          gamma -> c = V^{-1} gamma -> J in one call
//
// Cholesky kernels (row-major, lower triangle; the strictly upper triangle is
// never written), panels of 32 columns:
//   factor_diag  one CTA factors the 32 x 32 diagonal block, a row per lane
//   chol_trsm    rows below it: L21 = A21 L11^{-T}, a row per lane
//   chol_update  A22 -= L21 L21^T on 64 x 64 (few left: 32 x 32) tiles of the
//                lower triangle, the accumulators in registers (the FP64 pipe,
//                not shared memory or HBM, bounds this GEMM on GB300); the CTA
//                of the first tile goes on to factor the next diagonal block
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <memory>
#include <string>
#include <vector>

#include "../../include/lx3c.h"
#include "boys_device.cuh"
#include "lx3c_internal.h"

namespace lx3c {
cudaError_t launch_precompute(const DevBasis& orb, const int32_t* pairs, long long npair, int Ka, int Kb, double* rec,
                              double* ab, const DevBasis& aux, const int32_t* auxs, long long naux, int Kc,
                              double* auxrec, double* auxc, cudaStream_t st);
cudaError_t launch_eri3c(const ClassDesc& d, int grid, cudaStream_t st);
int eri3c_occupancy(int smem_bytes);
}  // namespace lx3c

using namespace lx3c;

namespace {

lx3c_status mfail(lx3c_status s, const std::string& m) {
  set_last_error(m);
  return s;
}

#define MCUDA(expr)                                                                                         \
  do {                                                                                                      \
    cudaError_t e_ = (expr);                                                                                \
    if (e_ != cudaSuccess) return mfail(LX3C_ECUDA, std::string(#expr) + ": " + cudaGetErrorString(e_));   \
  } while (0)

// Each of an SM's four sub-partitions issues one FP64 warp instruction per 64
// clocks, whether or not it depends on the last one (measured), so four warps
// share each serial part and every FP64 instruction of a column's chain
// counts: five for the reciprocal root, a product, an FMA.  32 columns take 12
// us (a 64-wide panel by one CTA with a root, a division and two block
// barriers per column took 110 us), and hide behind the update.  64 x 64 tiles
// replace 128 x 128 ones, which kept an SM busy for 250 us and left half the
// chip idle in matrices of a few thousand rows.
constexpr int kNB = 32;        // panel width of the Cholesky
constexpr int kSB = 64;        // block of the triangular solves

// ---------------------------------------------------------------------------
// Cholesky
// ---------------------------------------------------------------------------

struct CholMode {
  int* info;
  const double* diag0;  // drop mode: the original diagonal
  double drop_tol;
};

__device__ __forceinline__ bool is_zero(double x) {  // integer pipe: an FP64 compare costs 64 clocks
  return (__double2hiint(x) << 1 | __double2loint(x)) == 0;
}

// 1/sqrt of the pivot d of column g.  Dropped functions give 0 and a diagonal
// that is not positive gives NaN; d becomes the square of the factor's diagonal
// element in either case.
__device__ __forceinline__ double pivot_rsqrt(const CholMode& m, long long g, double& d, bool lead) {
  const int h = __double2hiint(d);
  if (m.diag0) {
    // drop mode: a pivot at or below drop_tol of the original diagonal marks
    // a function dependent on the earlier ones; an infinite pivot zeroes its
    // column below and its coefficient in the solves
    if (!(d > m.drop_tol * m.diag0[g])) {
      if (lead && m.info) ++*m.info;
      d = __longlong_as_double(0x7FF0000000000000LL);
      return 0.0;
    }
  }
  if (h > 0x38800000 && h < 0x47800000) return rsqrt_fp64(d);  // the range of its FP32 seed
  if (!(d > 0.0)) {  // not positive definite: record the first such pivot, carry NaN on
    if (lead && m.info && *m.info == 0) *m.info = (int)(g + 1);
    d = nan("");
  }
  return 1.0 / sqrt(d);
}

// Factor the nb x nb block at A[k][k] (nb <= 32) with 128 threads: lane i
// holds row i, warp w its columns w, w + 4, ...  The warp of the next column
// updates it first and publishes it before its other updates.
__device__ __forceinline__ void factor_diag(double* A, long long lda, long long k, int nb, const CholMode& mode,
                                            double (*s)[kNB + 1], double (*col)[kNB]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = warp; i < kNB; i += 4)
    s[i][lane] = i < nb && lane <= i ? A[(k + i) * lda + k + lane] : (i == lane ? 1.0 : 0.0);
  __syncthreads();
  double a[kNB / 4];
#pragma unroll
  for (int m = 0; m < kNB / 4; ++m) a[m] = s[lane][4 * m + warp];
  __syncthreads();
  const auto publish = [&](int j, double x) {
    double d = __shfl_sync(0xffffffffu, x, j);
    const double r = pivot_rsqrt(mode, k + j, d, lane == 0);
    const double v = lane > j && !is_zero(r) ? x * r : 0.0;
    col[j & 1][lane] = v;
    s[lane][j] = lane == j ? d : v;  // the diagonal's roots are taken together at the end
  };
  if (warp == 0 && nb > 0) publish(0, a[0]);
  __syncthreads();
#pragma unroll
  for (int j = 0; j + 1 < kNB; ++j) {
    if (j + 1 < nb) {
      // (entries above the diagonal pick up values that nothing reads)
      const double lj = -col[j & 1][lane];
      if (warp == ((j + 1) & 3)) publish(j + 1, fma(lj, col[j & 1][j + 1], a[(j + 1) >> 2]));
#pragma unroll
      for (int m = 0; m < kNB / 4; ++m) {
        const int c = 4 * m + warp;
        if (4 * m + 3 > j + 1 && c > j + 1) a[m] = fma(lj, col[j & 1][c], a[m]);
      }
      __syncthreads();
    }
  }
  if (warp == 0) s[lane][lane] = sqrt(s[lane][lane]);
  __syncthreads();
  for (int i = warp; i < nb; i += 4)
    if (lane <= i) A[(k + i) * lda + k + lane] = s[i][lane];
}

__global__ void __launch_bounds__(128) chol_diag(double* __restrict__ A, long long lda, int nb, CholMode mode) {
  __shared__ double s[kNB][kNB + 1];
  __shared__ double col[2][kNB];
  factor_diag(A, lda, 0, nb, mode, s, col);
}

// Rows k + nb + 16 blockIdx.x ... of the panel: x L11^T = a.  Warp w holds
// columns 8 w ... 8 w + 7 of the 16 rows, four per lane: each warp solves its
// columns in registers once the warps before it have published theirs.
constexpr int kTrsmRows = 16;

__global__ void __launch_bounds__(128) chol_trsm(double* __restrict__ A, long long lda, long long k, int nb,
                                                 long long n) {
  __shared__ double L[kNB][kNB + 1];
  __shared__ double X[kTrsmRows][kNB + 1];
  __shared__ double rd[kNB];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, row = lane & 15, half = lane >> 4;
  const long long r0 = k + nb + (long long)blockIdx.x * kTrsmRows;
#pragma unroll
  for (int i = warp; i < kNB; i += 4) L[i][lane] = i < nb && lane <= i ? A[(k + i) * lda + k + lane] : (i == lane ? 1.0 : 0.0);
#pragma unroll
  for (int r = warp; r < kTrsmRows; r += 4) X[r][lane] = r0 + r < n && lane < nb ? A[(r0 + r) * lda + k + lane] : 0.0;
  __syncthreads();
  if (warp == 0) rd[lane] = 1.0 / L[lane][lane];  // 0 for the infinite pivot of a dropped function
  double x[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) x[c] = X[row][8 * warp + 4 * half + c];
  __syncthreads();
  for (int w = 0; w < 4; ++w) {
    if (warp == w) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const double r = rd[8 * w + j];
        const double v = __shfl_sync(0xffffffffu, is_zero(r) ? 0.0 : x[j & 3] * r, row + 16 * (j >> 2));
        if (half == (j >> 2)) x[j & 3] = v;
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (4 + c > j && 4 * half + c > j) x[c] = fma(-v, L[8 * w + 4 * half + c][8 * w + j], x[c]);
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) X[row][8 * w + 4 * half + c] = x[c];
    }
    __syncthreads();
    if (warp > w) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const double v = X[row][8 * w + j];
#pragma unroll
        for (int c = 0; c < 4; ++c) x[c] = fma(-v, L[8 * warp + 4 * half + c][8 * w + j], x[c]);
      }
    }
  }
  for (int r = warp; r < kTrsmRows; r += 4)
    if (r0 + r < n && lane < nb) A[(r0 + r) * lda + k + lane] = X[r][lane];
}

// Lower tile (bi, bj), bj <= bi, of the trailing matrix (rows/cols from
// r0 = k + nb): A[i][j] -= sum_p L[i][k+p] L[j][k+p] for j <= i.  128 threads,
// (T/8) x (T/16) elements each.
template <int T>
__global__ void __launch_bounds__(128) chol_update(double* A, long long lda, long long k, int nb, long long n,
                                                   CholMode mode) {
  constexpr int RM = T / 8, CM = T / 16;
  __shared__ double As[kNB][T + 1], Bs[kNB][T + 1];  // rows of tiles bi and bj, transposed
  const long long x = blockIdx.x;
  long long bi = (long long)((sqrt(8.0 * (double)x + 1.0) - 1.0) * 0.5);
  while (bi * (bi + 1) / 2 > x) --bi;
  while ((bi + 1) * (bi + 2) / 2 <= x) ++bi;
  const long long bj = x - bi * (bi + 1) / 2;
  const long long r0 = k + nb, ri = r0 + bi * T, rj = r0 + bj * T;
  const int tid = threadIdx.x, p0 = tid & 31;
#pragma unroll 4
  for (int r = tid >> 5; r < T; r += 4) {
    As[p0][r] = ri + r < n && p0 < nb ? A[(ri + r) * lda + k + p0] : 0.0;
    Bs[p0][r] = rj + r < n && p0 < nb ? A[(rj + r) * lda + k + p0] : 0.0;
  }
  __syncthreads();
  const int ty = tid >> 4, tx = tid & 15;
  double acc[RM][CM];
#pragma unroll
  for (int r = 0; r < RM; ++r)
#pragma unroll
    for (int c = 0; c < CM; ++c) acc[r][c] = 0.0;
  for (int p = 0; p < nb; ++p) {
    double a[RM], b[CM];
#pragma unroll
    for (int r = 0; r < RM; ++r) a[r] = As[p][ty + 8 * r];
#pragma unroll
    for (int c = 0; c < CM; ++c) b[c] = Bs[p][tx + 16 * c];
#pragma unroll
    for (int r = 0; r < RM; ++r)
#pragma unroll
      for (int c = 0; c < CM; ++c) acc[r][c] = fma(a[r], b[c], acc[r][c]);
  }
#pragma unroll
  for (int r = 0; r < RM; ++r) {
    const long long i = ri + ty + 8 * r;
    if (i >= n) continue;
#pragma unroll
    for (int c = 0; c < CM; ++c) {
      const long long j = rj + tx + 16 * c;
      if (j <= i) A[i * lda + j] -= acc[r][c];
    }
  }
  if (x == 0) {
    __syncthreads();
    static_assert(T >= kNB, "the first tile holds the next diagonal block");
    factor_diag(A, lda, r0, (int)min((long long)kNB, n - r0), mode, (double (*)[kNB + 1])&As[0][0],
                (double (*)[kNB])&Bs[0][0]);
  }
}

// ---------------------------------------------------------------------------
// triangular solves, B row-major [n][nrhs], blocks of 64 rows
// ---------------------------------------------------------------------------

// Step of the solve for the block at k, with x the block solved before it (at
// kp, nbp rows; nbp = 0 for the first): the first CTAs subtract x's share from
// block k and solve it, kSolveCols right-hand sides each, the others subtract
// it from the rows still to come, which nothing else in the launch reads.  One
// launch per block: a separate diagonal solve by one thread per right-hand
// side took 60 us a block.  A CTA's eight warps take a column each, and more
// CTAs take the next eight: one CTA for all of them took 95.7 ms with 3,078
// functions and 256 right-hand sides, this 16.6 (8: 3.28 and 3.26).
// Forward: L x = b, rows descending; backward: L^T x = b, rows ascending.
constexpr int kSolveCols = 8;

template <bool kBack>
__global__ void __launch_bounds__(256) solve_step(const double* __restrict__ L, long long lda, long long k, int nb,
                                                  long long kp, int nbp, double* __restrict__ B, long long nrhs,
                                                  long long n) {
  __shared__ double s[kSB][kSB + 1];
  __shared__ double rd[kSB];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long ndiag = (nrhs + kSolveCols - 1) / kSolveCols;
  if (blockIdx.x >= ndiag) {
    if (!kBack) {
      // one warp per row, lanes over x's rows
      const long long i = k + nb + (blockIdx.x - ndiag) * 8 + warp;
      if (i >= n) return;
      const double l0 = lane < nbp ? L[i * lda + kp + lane] : 0.0;
      const double l1 = lane + 32 < nbp ? L[i * lda + kp + lane + 32] : 0.0;
      for (long long q = 0; q < nrhs; ++q) {
        double v = 0.0;
        if (lane < nbp) v = l0 * B[(kp + lane) * nrhs + q];
        if (lane + 32 < nbp) v = fma(l1, B[(kp + lane + 32) * nrhs + q], v);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) B[i * nrhs + q] -= v;
      }
    } else {
      // one thread per (row, right-hand side), reading a column of the block
      // row (coalesced across rows)
      const long long w = (blockIdx.x - ndiag) * 256 + tid;
      if (w >= k * nrhs) return;
      const long long j = w / nrhs, q = w - j * nrhs;
      double v0 = 0.0, v1 = 0.0;
      int i = 0;
      for (; i + 1 < nbp; i += 2) {
        v0 = fma(L[(kp + i) * lda + j], B[(kp + i) * nrhs + q], v0);
        v1 = fma(L[(kp + i + 1) * lda + j], B[(kp + i + 1) * nrhs + q], v1);
      }
      if (i < nbp) v0 = fma(L[(kp + i) * lda + j], B[(kp + i) * nrhs + q], v0);
      B[j * nrhs + q] -= v0 + v1;
    }
    return;
  }
  const long long c0 = (long long)blockIdx.x * kSolveCols;  // this CTA's columns
  const int nc = (int)min((long long)kSolveCols, nrhs - c0);
  // the diagonal block, kept in registers until the share is subtracted
  double dg[kSB * kSB / 256];
#pragma unroll
  for (int m = 0; m < kSB * kSB / 256; ++m) {
    const int idx = tid + 256 * m, i = idx / kSB, j = idx - i * kSB;
    dg[m] = i < nb && j <= i ? L[(k + i) * lda + k + j] : (i == j ? 1.0 : 0.0);
  }
  // x's share of block k (kBack: the transposed block below it)
  if (nbp > 0) {
    for (int idx = tid; idx < nb * nbp; idx += 256) {
      if (!kBack) {
        const int i = idx / nbp, p = idx - i * nbp;
        s[i][p] = L[(k + i) * lda + kp + p];
      } else {
        const int p = idx / nb, i = idx - p * nb;
        s[i][p] = L[(kp + p) * lda + k + i];
      }
    }
    __syncthreads();
    // four lanes per (row, right-hand side)
    const int part = tid & 3;
    for (int w0 = 0; w0 < nb * nc; w0 += 64) {
      const int w = w0 + (tid >> 2);
      const bool on = w < nb * nc;
      const int i = on ? w / nc : 0;
      const long long q = on ? c0 + w - i * nc : 0;
      double v0 = 0.0, v1 = 0.0;
      if (on)
#pragma unroll 4
        for (int p = part; p < nbp; p += 8) {
          v0 = fma(s[i][p], B[(kp + p) * nrhs + q], v0);
          if (p + 4 < nbp) v1 = fma(s[i][p + 4], B[(kp + p + 4) * nrhs + q], v1);
        }
      double v = v0 + v1;
      v += __shfl_xor_sync(0xffffffffu, v, 1);
      v += __shfl_xor_sync(0xffffffffu, v, 2);
      if (on && part == 0) B[(k + i) * nrhs + q] -= v;
    }
    __syncthreads();
  }
#pragma unroll
  for (int m = 0; m < kSB * kSB / 256; ++m) {
    const int idx = tid + 256 * m, i = idx / kSB, j = idx - i * kSB;
    if (kBack) s[j][i] = dg[m]; else s[i][j] = dg[m];
    if (i == j) rd[i] = 1.0 / dg[m];  // 0 for the infinite pivot of a dropped function
  }
  __syncthreads();
  // one warp per right-hand side, lane i holding rows i and i + 32
  if (warp < nc) {
    const long long q = c0 + warp;
    double b0 = lane < nb ? B[(k + lane) * nrhs + q] : 0.0;
    double b1 = lane + 32 < nb ? B[(k + lane + 32) * nrhs + q] : 0.0;
    // first the half whose unknowns come first, updating both, then the other
    double& f = kBack ? b1 : b0;
    double& g = kBack ? b0 : b1;
    const int of = kBack ? 32 : 0, og = 32 - of;
#pragma unroll 4
    for (int t = 0; t < 32; ++t) {
      const int j = kBack ? 31 - t : t;
      const double r = rd[of + j];
      const double xj = is_zero(r) ? 0.0 : __shfl_sync(0xffffffffu, f, j) * r;
      if (lane == j) f = xj;
      if (kBack ? lane < j : lane > j) f = fma(-s[of + lane][of + j], xj, f);
      g = fma(-s[og + lane][of + j], xj, g);
    }
#pragma unroll 4
    for (int t = 0; t < 32; ++t) {
      const int j = kBack ? 31 - t : t;
      const double r = rd[og + j];
      const double xj = is_zero(r) ? 0.0 : __shfl_sync(0xffffffffu, g, j) * r;
      if (lane == j) g = xj;
      if (kBack ? lane < j : lane > j) g = fma(-s[og + lane][og + j], xj, g);
    }
    if (lane < nb) B[(k + lane) * nrhs + q] = b0;
    if (lane + 32 < nb) B[(k + lane + 32) * nrhs + q] = b1;
  }
}

__global__ void copy_diag(const double* __restrict__ A, long long lda, long long n, double* __restrict__ d) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) d[i] = A[i * lda + i];
}

cudaError_t cholesky_launches(double* A, long long n, long long lda, int* info, const double* diag0,
                              double drop_tol, cudaStream_t st) {
  const CholMode mode{info, diag0, drop_tol};
  chol_diag<<<1, 128, 0, st>>>(A, lda, (int)std::min<long long>(kNB, n), mode);
  cudaError_t e = cudaGetLastError();
  for (long long k = 0; k + kNB < n && e == cudaSuccess; k += kNB) {
    const long long m = n - k - kNB;
    chol_trsm<<<(unsigned)((m + kTrsmRows - 1) / kTrsmRows), 128, 0, st>>>(A, lda, k, kNB, n);
    e = cudaGetLastError();
    if (e != cudaSuccess) continue;
    // 64 x 64 tiles while they fill the chip twice over, then 32 x 32 ones
    const long long t64 = (m + 63) / 64, t32 = (m + 31) / 32;
    if (t64 * (t64 + 1) / 2 >= 304)
      chol_update<64><<<(unsigned)(t64 * (t64 + 1) / 2), 128, 0, st>>>(A, lda, k, kNB, n, mode);
    else
      chol_update<32><<<(unsigned)(t32 * (t32 + 1) / 2), 128, 0, st>>>(A, lda, k, kNB, n, mode);
    e = cudaGetLastError();
  }
  return e;
}

cudaError_t solve_launches(const double* L, long long n, long long lda, double* B, long long nrhs, cudaStream_t st) {
  cudaError_t e = cudaSuccess;
  const long long ndiag = (nrhs + kSolveCols - 1) / kSolveCols;
  for (long long k = 0; k < n && e == cudaSuccess; k += kSB) {
    const int nb = (int)std::min<long long>(kSB, n - k);
    const long long rest = k > 0 ? n - k - nb : 0;
    solve_step<false><<<(unsigned)(ndiag + (rest + 7) / 8), 256, 0, st>>>(L, lda, k, nb, k - kSB, k > 0 ? kSB : 0, B, nrhs, n);
    e = cudaGetLastError();
  }
  const long long last = ((n - 1) / kSB) * kSB;
  for (long long k = last; k >= 0 && e == cudaSuccess; k -= kSB) {
    const int nb = (int)std::min<long long>(kSB, n - k);
    const int nbp = k == last ? 0 : (int)std::min<long long>(kSB, n - k - kSB);
    const long long rest = nbp > 0 ? k * nrhs : 0;
    solve_step<true><<<(unsigned)(ndiag + (rest + 255) / 256), 256, 0, st>>>(L, lda, k, nb, k + kSB, nbp, B, nrhs, n);
    e = cudaGetLastError();
  }
  return e;
}

}  // namespace

// ---------------------------------------------------------------------------
// metric plan
// ---------------------------------------------------------------------------

struct lx3c_metric {
  const lx3c_basis* aux = nullptr;
  lx3c_basis* bra = nullptr;  // the aux shells followed by the unit s shell (exponent 0)
  long long naux_ao = 0;
  struct Group {
    int l = 0, K = 0;
    std::vector<int> shells;
    int32_t* d_pairs = nullptr;   // (shell, unit shell)
    int32_t* d_kets = nullptr;
    int4* d_sub = nullptr;
    int* d_prim = nullptr;
    int4* d_pair_ao = nullptr;
    int* d_aux_ao = nullptr;
    double* d_pairrec = nullptr;
    double* d_pairab = nullptr;
    double* d_auxrec = nullptr;
    double* d_auxc = nullptr;
  };
  std::vector<Group> groups;
  struct Launch {
    ClassDesc desc;
    int grid = 1;
  };
  std::vector<Launch> launches;
  double flops = 0;
};

extern "C" {

void lx3c_metric_destroy(lx3c_metric* p) {
  if (!p) return;
  for (auto& g : p->groups) {
    cudaFree(g.d_pairs); cudaFree(g.d_kets); cudaFree(g.d_sub); cudaFree(g.d_prim); cudaFree(g.d_pair_ao);
    cudaFree(g.d_aux_ao); cudaFree(g.d_pairrec); cudaFree(g.d_pairab); cudaFree(g.d_auxrec); cudaFree(g.d_auxc);
  }
  lx3c_basis_destroy(p->bra);
  delete p;
}

lx3c_status lx3c_metric_plan(lx3c_metric** out, const lx3c_basis* aux, void* stream) {
  if (!out) return mfail(LX3C_EINVAL, "metric_plan: null output pointer");
  *out = nullptr;
  if (!aux || aux->nshell <= 0) return mfail(LX3C_EINVAL, "metric_plan: empty aux basis");
  for (int64_t s = 0; s < aux->nshell; ++s)
    if (aux->l[s] > LX3C_LMAX_AUX) return mfail(LX3C_ENOTSUP, "metric_plan: aux shell beyond the supported l");
  DevState* ds;
  int rc = device_state_get(&ds);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  std::unique_ptr<lx3c_metric, void (*)(lx3c_metric*)> p(new lx3c_metric, lx3c_metric_destroy);
  p->aux = aux;
  // bra basis: every aux shell, then the constant function 1 = exp(-0 r^2)
  lx3c_basis* b = new lx3c_basis;
  p->bra = b;
  b->nshell = aux->nshell + 1;
  b->nprim = aux->nprim + 1;
  b->l = aux->l; b->l.push_back(0);
  b->k = aux->k; b->k.push_back(1);
  b->atom = aux->atom; b->atom.push_back(-1);
  b->off = aux->off; b->off.push_back(aux->nprim);
  b->xyz = aux->xyz; b->xyz.insert(b->xyz.end(), {0.0, 0.0, 0.0});
  b->exps = aux->exps; b->exps.push_back(0.0);
  b->coefs = aux->coefs; b->coefs.push_back(1.0);
  rc = basis_upload(b, st);
  if (rc) return rc;
  const int unit = (int)aux->nshell;
  std::vector<int> aq(aux->nshell + 1, 0);
  for (int64_t s = 0; s < aux->nshell; ++s) aq[s + 1] = aq[s] + 2 * aux->l[s] + 1;
  p->naux_ao = aq[aux->nshell];
  std::map<std::pair<int, int>, std::vector<int>> byclass;
  for (int64_t s = 0; s < aux->nshell; ++s) byclass[{aux->l[s], aux->k[s]}].push_back((int)s);
  for (auto& kv : byclass) {
    lx3c_metric::Group g;
    g.l = kv.first.first;
    g.K = kv.first.second;
    g.shells = kv.second;
    const long long ns = (long long)g.shells.size();
    std::vector<int32_t> pairs(2 * ns);
    std::vector<int4> sub(ns), pao(ns);
    std::vector<int> prim(ns * g.K), aao(ns);
    for (long long i = 0; i < ns; ++i) {
      pairs[2 * i] = g.shells[i];
      pairs[2 * i + 1] = unit;
      sub[i] = int4{(int)i, (int)(i * g.K), g.K, 0};
      for (int r = 0; r < g.K; ++r) prim[i * g.K + r] = r;
      pao[i] = int4{aq[g.shells[i]], 0, 0, 0};
      aao[i] = aq[g.shells[i]];
    }
    MCUDA(cudaMalloc(&g.d_pairs, ns * 8));
    MCUDA(cudaMalloc(&g.d_kets, ns * 4));
    MCUDA(cudaMalloc(&g.d_sub, ns * sizeof(int4)));
    MCUDA(cudaMalloc(&g.d_prim, prim.size() * 4));
    MCUDA(cudaMalloc(&g.d_pair_ao, ns * sizeof(int4)));
    MCUDA(cudaMalloc(&g.d_aux_ao, ns * 4));
    MCUDA(cudaMalloc(&g.d_pairrec, (size_t)ns * g.K * kPairRec * 8));
    MCUDA(cudaMalloc(&g.d_pairab, (size_t)ns * 3 * 8));
    MCUDA(cudaMalloc(&g.d_auxrec, (size_t)ns * g.K * kAuxRec * 8));
    MCUDA(cudaMalloc(&g.d_auxc, (size_t)ns * 3 * 8));
    MCUDA(cudaMemcpyAsync(g.d_pairs, pairs.data(), ns * 8, cudaMemcpyHostToDevice, st));
    MCUDA(cudaMemcpyAsync(g.d_kets, g.shells.data(), ns * 4, cudaMemcpyHostToDevice, st));
    MCUDA(cudaMemcpyAsync(g.d_sub, sub.data(), ns * sizeof(int4), cudaMemcpyHostToDevice, st));
    MCUDA(cudaMemcpyAsync(g.d_prim, prim.data(), prim.size() * 4, cudaMemcpyHostToDevice, st));
    MCUDA(cudaMemcpyAsync(g.d_pair_ao, pao.data(), ns * sizeof(int4), cudaMemcpyHostToDevice, st));
    MCUDA(cudaMemcpyAsync(g.d_aux_ao, aao.data(), ns * 4, cudaMemcpyHostToDevice, st));
    p->groups.push_back(g);
  }
  // one class launch (lP 0 | lQ) per pair of groups
  for (auto& gp : p->groups)
    for (auto& gq : p->groups) {
      const ClassTables* ct;
      try {
        ct = &class_tables(gp.l, 0, gq.l, 1);
      } catch (std::exception& e) {
        return mfail(LX3C_ENOTSUP, std::string("metric_plan: ") + e.what());
      }
      DevClass* dc;
      rc = device_class_get(ds, *ct, &dc);
      if (rc) return rc;
      lx3c_metric::Launch L;
      ClassDesc& d = L.desc;
      const long long np = (long long)gp.shells.size(), nq = (long long)gq.shells.size();
      if (fill_class_desc(d, *ct, *dc, ds, 0, gp.K, gp.K, gq.K, nq) < 0)
        return mfail(LX3C_ENOTSUP, "metric_plan: class does not fit in shared memory");
      d.npair = np;
      d.naux = nq;
      d.nsub = np;
      d.ntile_aux = (int)((nq + d.T - 1) / d.T);
      d.ntiles = np * d.ntile_aux;
      d.subpairs = gp.d_sub;
      d.primidx = gp.d_prim;
      d.pairrec = gp.d_pairrec; d.pairab = gp.d_pairab;
      d.auxrec = gq.d_auxrec; d.auxc = gq.d_auxc;
      d.digest = 3;
      d.ldD = p->naux_ao;
      d.pair_ao = gp.d_pair_ao;
      d.aux_ao = gq.d_aux_ao;
      const int occ = eri3c_occupancy(d.smem_doubles * 8);
      L.grid = (int)std::min<long long>(d.ntiles, (long long)dev_nsm(ds) * occ * 8);
      double fl = 0;
      lx3c_class_flops(gp.l, 0, gq.l, gp.K, gq.K, 1, &fl);
      p->flops += fl * (double)np * (double)nq;
      p->launches.push_back(L);
    }
  MCUDA(cudaStreamSynchronize(st));
  *out = p.release();
  return LX3C_OK;
}

lx3c_status lx3c_metric_execute(lx3c_metric* p, double* V, void* stream) {
  if (!p || !V) return mfail(LX3C_EINVAL, "metric_execute: null pointer");
  cudaStream_t st = (cudaStream_t)stream;
  for (auto& g : p->groups) {
    const long long ns = (long long)g.shells.size();
    MCUDA(launch_precompute(p->bra->dev(), g.d_pairs, ns, g.K, 1, g.d_pairrec, g.d_pairab, p->aux->dev(), g.d_kets, ns,
                            g.K, g.d_auxrec, g.d_auxc, st));
  }
  for (auto& L : p->launches) {
    ClassDesc d = L.desc;
    d.out = V;
    MCUDA(launch_eri3c(d, L.grid, st));
  }
  return LX3C_OK;
}

lx3c_status lx3c_metric_info(const lx3c_metric* p, double* out, int n) {
  if (!p || (!out && n > 0)) return mfail(LX3C_EINVAL, "metric_info: null pointer");
  const double v[] = {(double)p->naux_ao, (double)p->groups.size(), (double)p->launches.size(),
                      1.0 * p->groups.size() + p->launches.size(), p->flops,
                      (double)p->aux->nshell * (double)p->aux->nshell};
  for (int i = 0; i < n && i < 6; ++i) out[i] = v[i];
  return LX3C_OK;
}

lx3c_status lx3c_cholesky(double* A, int64_t n, int64_t lda, double drop_tol, int32_t* info, void* stream) {
  if (!A || n < 1 || lda < n) return mfail(LX3C_EINVAL, "cholesky: null matrix, n < 1 or lda < n");
  if (!(drop_tol >= 0.0 && drop_tol < 1.0)) return mfail(LX3C_EINVAL, "cholesky: drop_tol must be in [0, 1)");
  cudaStream_t st = (cudaStream_t)stream;
  if (info) MCUDA(cudaMemsetAsync(info, 0, sizeof(int32_t), st));
  double* diag0 = nullptr;
  if (drop_tol > 0.0) {
    MCUDA(cudaMallocAsync(&diag0, (size_t)n * sizeof(double), st));
    copy_diag<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(A, lda, n, diag0);
    MCUDA(cudaGetLastError());
  }
  cudaError_t e = cholesky_launches(A, n, lda, info, diag0, drop_tol, st);
  if (diag0) cudaFreeAsync(diag0, st);
  MCUDA(e);
  return LX3C_OK;
}

lx3c_status lx3c_cholesky_solve(const double* L, int64_t n, int64_t lda, double* B, int64_t nrhs, void* stream) {
  if (!L || !B || n < 1 || lda < n || nrhs < 1) return mfail(LX3C_EINVAL, "cholesky_solve: bad argument");
  MCUDA(solve_launches(L, n, lda, B, nrhs, (cudaStream_t)stream));
  return LX3C_OK;
}

lx3c_status lx3c_dfj_coulomb(lx3c_dfj* plan, const double* L, int64_t lda, const double* D, double* gamma,
                             double* c, double* J, void* stream) {
  if (!plan || !L || !D || !gamma || !c || !J) return mfail(LX3C_EINVAL, "dfj_coulomb: null pointer");
  double info[7];
  lx3c_status rc = lx3c_dfj_info(plan, info, 7);
  if (rc) return rc;
  const long long naux_ao = (long long)info[6];
  if (lda < naux_ao) return mfail(LX3C_EINVAL, "dfj_coulomb: lda smaller than the aux AO count");
  cudaStream_t st = (cudaStream_t)stream;
  rc = lx3c_dfj_execute(plan, D, c, gamma, nullptr, stream);  // gamma only; c is not read
  if (rc) return rc;
  MCUDA(cudaMemcpyAsync(c, gamma, naux_ao * sizeof(double), cudaMemcpyDeviceToDevice, st));
  MCUDA(solve_launches(L, naux_ao, lda, c, 1, st));
  return lx3c_dfj_execute(plan, D, c, nullptr, J, stream);
}

}  // extern "C"
