// FP32 passes of the 1152 x 1152 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(1152)
}  // namespace qg
