// Hermite-density path of the DF-J build and its gradient (hermite.cu):
// plan of one (orbital basis, auxiliary basis) pair and its launches.
#pragma once
#include <cuda_runtime.h>

#include <string>
#include <vector>

#include "lx3c_internal.h"

namespace lx3c {

// Shell pairs of one bra class, in the caller's canonical order.
struct HermBra {
  int la, lb, Ka, Kb;
  std::vector<int32_t> pairs;  // [n][2]
  std::vector<double> q;       // screening factor of each pair (unscaled)
  double nprim;                // contributing primitive pairs of a pair, on average
};

// Ket shells of one (lc, Kc), sorted by decreasing screening factor.
struct HermKet {
  int lc, Kc;
  std::vector<int32_t> shells;
  std::vector<double> q;
};

struct HermPlan;

// Number of kets of the sorted list that a pair of factor q keeps.
typedef int (*HermKeep)(double qpair, const std::vector<double>& qket, double tol);

// Build the plan for the (bra, ket) classes where use(bra, ket) holds.  grad:
// energy gradient (programs one Hermite degree higher).  Returns an lx3c_status.
int herm_build(HermPlan** out, const lx3c_basis* orb, const lx3c_basis* aux, const std::vector<HermBra>& bras,
               const std::vector<HermKet>& kets, bool (*use)(const HermBra&, const HermKet&), HermKeep keep, double tol,
               bool grad, long long nao, cudaStream_t st);
void herm_destroy(HermPlan* p);
// gamma (gacc) and J (Jacc) into the fixed-point accumulators; either may be null.
cudaError_t herm_execute(HermPlan* p, const double* D, const double* c, unsigned long long* gacc,
                         unsigned long long* Jacc, cudaStream_t st);
// dE/dR of E = c^T gamma into the fixed-point accumulators facc [natom][3].
cudaError_t herm_gradient(HermPlan* p, const double* D, const double* c, unsigned long long* facc, cudaStream_t st);
int herm_launches(const HermPlan* p);       // kernels of one execute (or gradient)
double herm_flops(const HermPlan* p);       // FP64 flops of one fused execute (or gradient)
double herm_class_flops(int Lab, int lc);   // per primitive triple, gamma and J fused
double herm_max_adds(const HermPlan* p);    // upper bound of the additions into one gradient accumulator

}  // namespace lx3c
