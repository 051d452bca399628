// FP32 passes of the 1458 x 1458 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(1458)
}  // namespace qg
