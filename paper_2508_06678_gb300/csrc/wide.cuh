// The row and column passes of row_kernel.cuh / column_kernel.cuh with the transform's length fixed at compile time.
// Included by the grid_<N>.cu of the small FP32 grids, one translation unit per grid size.
#pragma once

#include "column_kernel.cuh"
#include "row_kernel.cuh"

namespace qg {

template <int N>
cudaError_t launch_row_wide(const Geom& g, const FftPlan& plan, const RowDesc& d, const void* tw, cudaStream_t st) {
  return launch_row_shape<float>(g, plan, StShape<N, fft_elems(N)>{}, d, tw, st);
}
template <int N>
cudaError_t launch_col_wide(const Geom& g, const FftPlan& plan, const ColDesc& d, const void* tw, int W,
                            cudaStream_t st) {
  return launch_col_shape<float>(g, plan, StShape<N, fft_elems(N)>{}, d, tw, W, st);
}

#define QG_INSTANTIATE_WIDE(N)                                                                                    \
  template cudaError_t launch_row_wide<N>(const Geom&, const FftPlan&, const RowDesc&, const void*, cudaStream_t); \
  template cudaError_t launch_col_wide<N>(const Geom&, const FftPlan&, const ColDesc&, const void*, int, cudaStream_t);

}  // namespace qg
