// FP32 passes of the 1024 x 1024 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(1024)
}  // namespace qg
