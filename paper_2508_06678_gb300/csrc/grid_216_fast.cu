// FP32 passes of the 216 x 216 grid, one transform after another; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(216)
}  // namespace qg
