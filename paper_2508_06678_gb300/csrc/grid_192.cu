// FP32 passes of the 192 x 192 grid; see wide.cuh.
#include "wide.cuh"

namespace qg {
QG_INSTANTIATE_WIDE(192)
}  // namespace qg
