// FP32 passes of the 2304 x 2304 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(2304)
}  // namespace qg
