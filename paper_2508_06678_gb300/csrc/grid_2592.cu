// FP32 passes of the 2592 x 2592 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(2592)
}  // namespace qg
