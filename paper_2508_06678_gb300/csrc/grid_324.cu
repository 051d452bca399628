// FP32 passes of the 324 x 324 grid; see wide.cuh.
#include "wide.cuh"

namespace qg {
QG_INSTANTIATE_WIDE(324)
}  // namespace qg
