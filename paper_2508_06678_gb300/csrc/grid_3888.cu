// FP32 passes of the 3888 x 3888 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(3888)
}  // namespace qg
