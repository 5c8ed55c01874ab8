// Data and device code that the table-driven and the unrolled Hermite kernels
// (hermite.cu, hermite_unrolled.cu) share.
#pragma once
#include <cuda_runtime.h>

#include "fixed128.cuh"
#include "lx3c_internal.h"

namespace lx3c {

constexpr int kMaxDeg = 13;  // Hermite degrees 0..13 (la + lb <= 12, one more for the gradient)
constexpr unsigned kLast = 0x80000000u;
constexpr int kColBytes = 32 * 8;  // one column: a double per lane

__host__ __device__ constexpr int nherm(int L) { return (L + 1) * (L + 2) * (L + 3) / 6; }
// position of (x, y, z) in the graded Hermite order
__host__ __device__ constexpr int hidx(int x, int y, int z) {
  const int n = x + y + z, m = y + z;
  return n * (n + 1) * (n + 2) / 6 + m * (m + 1) / 2 + z;
}

// A list of outputs, each a sum of products of two columns.  Four queues of
// outputs run side by side, balanced in length: a batch is one term of each
// queue, the two factors as byte offsets in a and b; the sign bit of a queue's
// b closes its output, whose header word (destination byte offset | palette id
// of its scale factor << 20; for y rows Hermite index | axes << 16) is the next
// of h.  The queues' ragged ends multiply the zero column.
// Each warp of the block has queues of its own: nb + 1 batches and hs headers
// on from the one before.
struct Stage {
  const uint4* a;
  const uint4* b;
  const unsigned* h;
  int nb;  // even
  int hs;
};

struct HermCls {
  int nw;  // warps per block
  int Lab, lc, Kc, L, nR, nY, ncc, nC, W, nket;
  int cX, cPW, cU, cB, cCP, cGA;  // column offsets (R at column 0)
  int cZero, cH;          // the zero column; the primitive pairs' densities
  int rbeg[kMaxDeg + 2];  // R recursion: operations of level m at rops[rbeg[m]] ...
  const uint4* rops;
  Stage Z, gz, gy, gx;    // gamma: Z_u, then the shift's transpose along z, y, x
  Stage jx, jy, jw;       // J: the shift of q along x, y, z
  Stage Y;                // y_a
  const int* cptr;        // Cartesian c -> (C, T_Cc c!) and its transpose
  const int2* cent;
  const int* gptr;
  const int2* gent;
  const double* pal;
  const int* ydeg;        // degree of Hermite index a
  double boys_cL;
  // data
  const double* prim;     // [nprim][4]: gamma, P
  const double* scale;    // [nprim][2][Lab + 1]: factor of y_a by degree, power of two it holds (inverse)
  const int* primpair;    // primitive -> pair position
  const int* cnt;         // kets kept by each pair
  const double* H;        // [nprim][nR], gradient: [nprim][3][nY]
  unsigned long long* Yacc;
  const double* auxrec;   // [nket][Kc][2]
  const double* auxc;     // [nket][3]
  const int* aux_ao;
  const int* aux_atom;
};

struct HermArgs {
  const HermCls* cls;
  const int4* tiles;  // {class, first ket, first primitive, primitives}
  const double* boys_tab;
  const double* boys_mid;
  const double* cvec;
  unsigned long long* gacc;
  unsigned long long* facc;
};

// Adds to y the sums over kets of `row` staged rows of 32 lanes (row stride
// 33): 32 / rows lanes per row, a power of two, sum the W kets of each of the
// 32 / W primitive pairs.  index(r): the Hermite index of staged row r.
template <class Ix>
__device__ __forceinline__ void sum_rows(const HermCls& c, const double* stg, int row, const int4& tile, int e0,
                                         int lane, const Ix& index) {
  const int W = c.W;
  __syncwarp();
  const int lg = row > 16 ? 0 : (row > 8 ? 1 : (row > 4 ? 2 : (row > 2 ? 3 : (row > 1 ? 4 : 5))));
  const int w = 32 >> lg, r = lane >> lg, part = lane & ((1 << lg) - 1);
  const int a = index(r);
  const int seg = min(w, W);  // kets summed by this lane for one primitive pair
  const double* x = stg + r * 33 + part * w;
  for (int s0 = 0; s0 < w; s0 += seg) {
    double v0 = 0.0, v1 = 0.0;
    if (r < row) {
      int i = 0;
      for (; i + 1 < seg; i += 2) {
        v0 += x[s0 + i];
        v1 += x[s0 + i + 1];
      }
      if (i < seg) v0 += x[s0 + i];
    }
    double v = seg > 1 ? v0 + v1 : v0;
    for (int o = 1; o * w < W; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int at = part * w + s0, s = at / W;
    if (r < row && at == s * W && e0 + s < tile.w) {
      const int ps = tile.z + e0 + s;
      v *= __ldg(c.scale + 2LL * ps * (c.Lab + 1) + __ldg(c.ydeg + a));
      wide_add(c.Yacc + kWideWords * ((long long)ps * c.nY + a), v);
    }
  }
  __syncwarp();
}

// Classes (Lab, lc) of the unrolled kernel: up to degree 6, as far as the
// shared-memory columns let five or more one-warp blocks onto an SM.  (l s|C)
// classes below lc = 5 belong to the register kernels of eri3c.cu.
__host__ __device__ constexpr bool herm_unrolled(int Lab, int lc) {
  return lc <= 6 && (Lab == 1 ? lc >= 5 : Lab >= 2 && Lab <= 6 && lc <= (Lab < 5 ? 6 : 5));
}
__host__ __device__ constexpr bool unrolled_m_shared(int Lab, int lc) { return Lab >= 5 || lc == 6 || Lab + lc >= 9; }
template <int Lab>
cudaError_t herm_unrolled_setup();
template <int Lab>
cudaError_t herm_unrolled_launch(const HermArgs& a, int mode, int smem, long long n, cudaStream_t st);
struct UnrolledCost {
  double base, gamma, j;  // FP64 instructions per primitive triple
};
UnrolledCost herm_unrolled_cost(int Lab, int lc);
int herm_unrolled_smem(int Lab, int lc, int W);  // bytes
// mode: bit 0 gamma, bit 1 J, 4 gradient; n tiles, all of classes with this Lab
cudaError_t launch_herm_unrolled(int Lab, const HermArgs& a, int mode, int smem, long long n, cudaStream_t st);
cudaError_t herm_unrolled_setup();

}  // namespace lx3c
