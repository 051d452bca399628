// FP64 instances of the row pass.
#include "row_kernel.cuh"

namespace qg {
template cudaError_t launch_row<double>(const Geom&, const FftPlan&, const RowDesc&, const void*, cudaStream_t);
}
