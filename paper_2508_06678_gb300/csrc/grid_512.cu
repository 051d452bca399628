// FP32 passes of the 512 x 512 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(512)
}  // namespace qg
