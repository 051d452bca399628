// FP32 instances of the column pass.
#include "column_kernel.cuh"

namespace qg {
template cudaError_t launch_col<float>(const Geom&, const FftPlan&, const ColDesc&, const void*, int, cudaStream_t);
}
