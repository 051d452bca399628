// FP32 passes of the 1944 x 1944 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(1944)
}  // namespace qg
