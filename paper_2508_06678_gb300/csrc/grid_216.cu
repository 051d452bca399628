// FP32 passes of the 216 x 216 grid; see wide.cuh.
#include "wide.cuh"

namespace qg {
QG_INSTANTIATE_WIDE(216)
}  // namespace qg
