// FP32 passes of the 768 x 768 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(768)
}  // namespace qg
