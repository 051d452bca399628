// FP32 passes of the 576 x 576 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(576)
}  // namespace qg
