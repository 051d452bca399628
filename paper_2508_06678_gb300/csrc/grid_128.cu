// FP32 passes of the 128 x 128 grid; see wide.cuh.
#include "wide.cuh"

namespace qg {
QG_INSTANTIATE_WIDE(128)
}  // namespace qg
