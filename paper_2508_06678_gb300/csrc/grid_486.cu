// FP32 passes of the 486 x 486 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(486)
}  // namespace qg
