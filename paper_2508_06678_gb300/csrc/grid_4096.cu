// FP32 passes of the 4096 x 4096 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(4096)
}  // namespace qg
