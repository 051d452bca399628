// FP32 passes of the 1728 x 1728 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(1728)
}  // namespace qg
