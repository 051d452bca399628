// FP32 passes of the 1536 x 1536 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(1536)
}  // namespace qg
