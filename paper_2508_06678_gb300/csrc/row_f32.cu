// FP32 instances of the row pass.
#include "row_kernel.cuh"

namespace qg {
template cudaError_t launch_row<float>(const Geom&, const FftPlan&, const RowDesc&, const void*, cudaStream_t);
}
