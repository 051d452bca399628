// FP32 passes of the 288 x 288 grid, one transform after another; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(288)
}  // namespace qg
