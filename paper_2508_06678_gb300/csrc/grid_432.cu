// FP32 passes of the 432 x 432 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(432)
}  // namespace qg
