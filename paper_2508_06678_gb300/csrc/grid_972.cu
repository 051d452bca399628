// FP32 passes of the 972 x 972 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(972)
}  // namespace qg
