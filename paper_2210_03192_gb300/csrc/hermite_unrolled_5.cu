// The unrolled Hermite kernel of degree 5.
#include "hermite_unrolled.cuh"

namespace lx3c {

LX3C_HERM_UNROLLED(5)

}  // namespace lx3c
