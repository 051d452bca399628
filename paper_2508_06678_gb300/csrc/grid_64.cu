// FP32 passes of the 64 x 64 grid; see wide.cuh.
#include "wide.cuh"

namespace qg {
QG_INSTANTIATE_WIDE(64)
}  // namespace qg
