// Host side of the unrolled Hermite kernels: their cost and shared memory, and
// the kernels of degree 1, 2 and 6 (the others are compiled beside, for the
// build's time).
#include <algorithm>

#include "hermite_unrolled.cuh"

namespace lx3c {

LX3C_HERM_UNROLLED(1)
LX3C_HERM_UNROLLED(2)
LX3C_HERM_UNROLLED(6)

int herm_unrolled_smem(int Lab, int lc, int W) {
  const int NR = nherm(Lab), ncc = (lc + 1) * (lc + 2) / 2, NU = nherm(std::min(Lab, lc));
  const int nm = unrolled_m_shared(Lab, lc) ? (nherm(lc) - nherm(lc - std::min(Lab, lc) - 1)) * 32 : 0;
  return ((32 / W * NR + 31) / 32 * 32 + (ncc + NU) * 32 + std::max(nm, std::min(NR, kRowsMost) * 33)) * 8;
}

static UnrolledCost count(int Lab, int lc) {
  UnrolledCost k;
  k.base = 40 + 8 + 4.0 * Lab + std::max(0, nherm(lc) - 4);
  for (int m = 0; m < Lab; ++m)
    for (int h = 1; h < nherm(Lab - m); ++h) k.base += power(h) == 1 ? 1 : 2;
  double shift = 0, conv = 0;  // X_u or G_c; Z_u or y_a
  for (int u = 0; u < nherm(std::min(Lab, lc)); ++u) {
    const int n = lc - deg(u);
    shift += (n + 1) * (n + 2) / 2 + (fact3(u) != 1.0);
    conv += nherm(Lab - deg(u));
  }
  k.gamma = conv + shift;
  k.j = conv + shift + 1.2 * nherm(Lab);
  return k;
}

UnrolledCost herm_unrolled_cost(int Lab, int lc) {
  struct Table {
    UnrolledCost k[7][7];
    Table() {
      for (int L = 1; L < 7; ++L)
        for (int l = 0; l < 7; ++l) k[L][l] = count(L, l);
    }
  };
  static const Table t;
  return t.k[Lab][lc];
}

cudaError_t herm_unrolled_setup() {
  cudaError_t e = herm_unrolled_setup<1>();
  if (e == cudaSuccess) e = herm_unrolled_setup<2>();
  if (e == cudaSuccess) e = herm_unrolled_setup<3>();
  if (e == cudaSuccess) e = herm_unrolled_setup<4>();
  if (e == cudaSuccess) e = herm_unrolled_setup<5>();
  if (e == cudaSuccess) e = herm_unrolled_setup<6>();
  return e;
}

cudaError_t launch_herm_unrolled(int Lab, const HermArgs& a, int mode, int smem, long long n, cudaStream_t st) {
  switch (Lab) {
    case 1: return herm_unrolled_launch<1>(a, mode, smem, n, st);
    case 2: return herm_unrolled_launch<2>(a, mode, smem, n, st);
    case 3: return herm_unrolled_launch<3>(a, mode, smem, n, st);
    case 4: return herm_unrolled_launch<4>(a, mode, smem, n, st);
    case 5: return herm_unrolled_launch<5>(a, mode, smem, n, st);
    case 6: return herm_unrolled_launch<6>(a, mode, smem, n, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lx3c
