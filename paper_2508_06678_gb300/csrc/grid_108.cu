// FP32 passes of the 108 x 108 grid; see wide.cuh.
#include "wide.cuh"

namespace qg {
QG_INSTANTIATE_WIDE(108)
}  // namespace qg
