// FP32 passes of the 288 x 288 grid; see wide.cuh.
#include "wide.cuh"

namespace qg {
QG_INSTANTIATE_WIDE(288)
}  // namespace qg
