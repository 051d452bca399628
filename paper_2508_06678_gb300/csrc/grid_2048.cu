// FP32 passes of the 2048 x 2048 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(2048)
}  // namespace qg
