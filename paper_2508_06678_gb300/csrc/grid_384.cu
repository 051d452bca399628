// FP32 passes of the 384 x 384 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(384)
}  // namespace qg
