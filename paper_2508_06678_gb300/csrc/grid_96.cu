// FP32 passes of the 96 x 96 grid; see wide.cuh.
#include "wide.cuh"

namespace qg {
QG_INSTANTIATE_WIDE(96)
}  // namespace qg
