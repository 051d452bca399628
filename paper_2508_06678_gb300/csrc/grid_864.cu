// FP32 passes of the 864 x 864 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(864)
}  // namespace qg
