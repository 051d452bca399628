// FP32 passes of the 256 x 256 grid, one transform after another; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(256)
}  // namespace qg
