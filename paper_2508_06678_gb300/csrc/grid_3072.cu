// FP32 passes of the 3072 x 3072 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(3072)
}  // namespace qg
