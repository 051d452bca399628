// The compile-time engine of the large FP32 grids' row and column passes (fast_kernels.cuh).
//
// Plan, ownership and twiddle tables are those of fft.cuh: a length-N sequence is owned by TT = N / EL threads,
// thread t holding the EL elements t + TT m; every pass reads the thread's own elements and the last pass lands on
// them again.  Hence an inverse FFT, any pointwise work and a forward FFT chain with no shared-memory traffic between
// them, and every column-pass spectral operation happens in registers on the thread's own k values.  Shared memory
// is padded by one element every 16 so the exchanges are free of bank conflicts.
#pragma once

#include "fft.cuh"
#include "qg_common.cuh"

namespace qg {
namespace fast {

template <typename T, int N> struct Eng {
  using C = cplx_t<T>;
  static constexpr int EL = fft_elems(N);
  static constexpr int TT = N / EL;
  static constexpr Radices P = fft_radices(N, EL);
  static constexpr int NEX = P.np - 1;    // shared-memory exchanges of one transform
  static constexpr int BUF = N + N / 16 + (N % 16 ? 1 : 0);  // padded complex elements of one sequence
  static constexpr int K = (N - 1) / 3;
  static constexpr int Kc = K + 1;

  __device__ static __forceinline__ int pad(int i) { return fft_pad(i); }

  template <int I, bool PK>
  __device__ static __forceinline__ void from(C* x, int t, C* b0, C* b1, int& ph, const C* __restrict__ ptw, int sign,
                                              bool active) {
    if constexpr (I < P.np) {
      C* buf = ph ? b1 : b0;
      st_pass<C, N, EL, I, PK, true>(x, t, buf, ptw, sign, active, BUF, nullptr);
      if constexpr (I < P.np - 1) {
        __syncthreads();
#pragma unroll
        for (int m = 0; m < EL; ++m) x[m] = buf[pad(t + TT * m)];
        ph ^= 1;
        from<I + 1, PK>(x, t, b0, b1, ph, ptw, sign, active);
      }
    }
  }

  // Full transform.  b0, b1 alternate per exchange (ph toggles); callers pass the same ph through every use of the
  // two buffers.  PK: packed FP32 butterflies (QG_PACKED_F32).  Threads that are not active only keep the barriers.
  template <bool PK = true>
  __device__ static __forceinline__ void run(C* x, int t, C* b0, C* b1, int& ph, const C* __restrict__ ptw, int sign,
                                             bool active = true) {
    from<0, PK>(x, t, b0, b1, ph, ptw, sign, active);
  }
};

}  // namespace fast

// rows of one TMA box of the specialised column pass: N split evenly into boxes of at most 256 rows (a multiple of 8,
// so that every box starts on 128 bytes of shared memory); the last box may reach past the array, where loads read
// zeros and stores are dropped
constexpr int fast_box_rows(int n) {
  const int nbox = (n + 255) / 256;
  return ((n + nbox - 1) / nbox + 7) / 8 * 8;
}

// k_x columns per CTA of the specialised column pass
constexpr int kFastWidth = 2;
template <typename T, int N>
cudaError_t launch_row_fast(const Geom& g, const RowDesc& d, const void* tw, cudaStream_t st);
struct TmaSet;
template <typename T, int N>
cudaError_t launch_col_fast(const Geom& g, const ColDesc& d, const void* tw, const TmaSet& tm, cudaStream_t st);

}  // namespace qg
