// FP32 passes of the 324 x 324 grid, one transform after another; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(324)
}  // namespace qg
