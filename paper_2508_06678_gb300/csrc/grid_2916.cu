// FP32 passes of the 2916 x 2916 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(2916)
}  // namespace qg
