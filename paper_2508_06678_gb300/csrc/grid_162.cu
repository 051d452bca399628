// FP32 passes of the 162 x 162 grid; see wide.cuh.
#include "wide.cuh"

namespace qg {
QG_INSTANTIATE_WIDE(162)
}  // namespace qg
