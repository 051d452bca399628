// FP32 passes of the 192 x 192 grid, one transform after another; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(192)
}  // namespace qg
