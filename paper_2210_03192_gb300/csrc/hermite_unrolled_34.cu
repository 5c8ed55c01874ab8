// The unrolled Hermite kernels of degree 3 and 4.
#include "hermite_unrolled.cuh"

namespace lx3c {

LX3C_HERM_UNROLLED(3)
LX3C_HERM_UNROLLED(4)

}  // namespace lx3c
