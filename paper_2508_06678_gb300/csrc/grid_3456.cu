// FP32 passes of the 3456 x 3456 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(3456)
}  // namespace qg
