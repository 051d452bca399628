// FP32 passes of the 72 x 72 grid; see wide.cuh.
#include "wide.cuh"

namespace qg {
QG_INSTANTIATE_WIDE(72)
}  // namespace qg
