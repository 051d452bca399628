// FP32 passes of the 256 x 256 grid; see wide.cuh.
#include "wide.cuh"

namespace qg {
QG_INSTANTIATE_WIDE(256)
}  // namespace qg
