// FP32 passes of the 648 x 648 grid; see fast_kernels.cuh.
#include "fast_kernels.cuh"

namespace qg {
QG_INSTANTIATE_FAST(648)
}  // namespace qg
