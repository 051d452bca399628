// FP32 passes of the 1296 x 1296 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(1296)
}  // namespace qg
