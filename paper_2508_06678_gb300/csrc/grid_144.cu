// FP32 passes of the 144 x 144 grid; see wide.cuh.
#include "wide.cuh"

namespace qg {
QG_INSTANTIATE_WIDE(144)
}  // namespace qg
