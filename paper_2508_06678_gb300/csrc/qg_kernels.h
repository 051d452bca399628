// Host-side declarations of the kernel launchers of libqg.
#pragma once

#include "fft.cuh"

namespace qg {

// SMs of the current device, queried once per device (concurrent first calls store the same value)
int device_sms();

// Launch shape of the row pass: rows per CTA, groups (transforms side by side), physical rows kept in shared memory
// per row (slots).
// (the first `full` CTAs have `rows` rows, the others one)
struct RowConfig {
  int full, rows, groups, threads, nslot, one_buf, warp;
  size_t smem;
};
RowConfig row_config(const FftPlan& p, const RowDesc& d, int esz);
template <typename T>
cudaError_t launch_row(const Geom& g, const FftPlan& plan, const RowDesc& d, const void* tw, cudaStream_t st);

// Launch shape of the column pass: w columns per CTA, fields transformed side by side, buffer pitch.
// The first `full` CTAs do a column's work alone; each of the other columns has `split` CTAs, which all transform its
// incoming fields and each derive a part of the outgoing ones.
struct ColConfig {
  int full, split, grid, w, fields, threads, pitch, one_buf, warp;
  size_t smem;
};
ColConfig col_config(const Geom& g, const FftPlan& p, const ColDesc& d, int W, int esz);
template <typename T>
cudaError_t launch_col(const Geom& g, const FftPlan& plan, const ColDesc& d, const void* tw, int W, cudaStream_t st);
// columns per CTA of the column pass (the mixed arrays' pitch is a multiple of it)
int col_width(const FftPlan& p, int esz);

// FP32 grids with passes specialised for N (grid_<N>.cu): transforms side by side (wide) or one after another (fast).
// Side by side pays while a grid leaves SMs idle and a row has enough transforms to fill them, so the dynamic closures'
// up to 324, the others' below 192.  Measured, us per step side by side / one after another: Leith 256^2 60 / 58,
// 324^2 108 / 94, 512^2 96 / 68; dynamic Smagorinsky 192^2 102 / 140, 256^2 89 / 105, 324^2 169 / 210, 384^2 152 / 145.
#define QG_WIDE_GRIDS(X) X(64) X(72) X(96) X(108) X(128) X(144) X(162) X(192) X(216) X(256) X(288) X(324)
#define QG_FAST_GRIDS(X)                                                                         \
  X(192) X(216) X(256) X(288) X(324) X(384) X(432) X(486) X(512) X(576) X(648) X(768) X(864) X(972) X(1024) X(1152) X(1296) \
  X(1458) X(1536) X(1728) X(1944) X(2048) X(2304) X(2592) X(2916) X(3072) X(3456) X(3888) X(4096)
#define X(N) || n == N
constexpr bool wide_grid(int n) { return false QG_WIDE_GRIDS(X); }
constexpr bool fast_grid(int n) { return false QG_FAST_GRIDS(X); }
#undef X
template <int N>
cudaError_t launch_row_wide(const Geom& g, const FftPlan& plan, const RowDesc& d, const void* tw, cudaStream_t st);
template <int N>
cudaError_t launch_col_wide(const Geom& g, const FftPlan& plan, const ColDesc& d, const void* tw, int W,
                            cudaStream_t st);

// Spectral diagnostics: out[0] = sum w |k|^2 |psi|^2, out[1] = sum w |w|^2 over the stored half spectrum
// (w = 1 on the k_x = 0 column, else 2), FP64, deterministic two-level reduction.
template <typename T>
cudaError_t launch_spectral_sums(const Geom& g, const void* w0, double* partials, int nblk, double* out,
                                 cudaStream_t st);

// Physical max |f| and finiteness: out[0] = max |f|, out[1] = 1 if all finite else 0.
template <typename T>
cudaError_t launch_phys_maxabs(const Geom& g, const void* f, double* partials, int nblk, double* out,
                               cudaStream_t st);

// ---- discrete adjoint of the step (adjoint.cu)
// spectral multipliers of adj_combine (conjugates are the transposes the adjoint needs)
enum AdjMul : int {
  AM_ONE = 0,
  AM_CU,    // -i k_y / |k|^2   transpose of w -> u
  AM_CV,    // +i k_x / |k|^2   transpose of w -> v
  AM_CX,    // -i k_x           transpose of d/dx
  AM_CY,    // -i k_y           transpose of d/dy
  AM_IX,    // +i k_x
  AM_IY,    // +i k_y
  AM_XY,    // k_x k_y / |k|^2           w -> psi_xy
  AM_DD,    // (k_x^2 - k_y^2) / |k|^2   w -> psi_xx - psi_yy
  AM_VISC,  // exp(-(nu |k|^2 + mu) dt)
};
constexpr int AM_TESTF = 0x100;  // flag: also multiply by the test filter, |m|^2 (2r)^2 <= N^2
constexpr int kAdjTerms = 12;
struct AdjTerm {
  const void* in;        // spectral array (stored band layout)
  int code;              // AdjMul, optionally | AM_TESTF
  double coef;
  const double* cptr;    // if set, coef is multiplied by this device scalar
};
struct AdjCombine {
  void* out;
  int accumulate;  // out += sum (else out = sum)
  int zero_mean;   // set the (0, 0) mode to zero
  int nterm;
  AdjTerm term[kAdjTerms];
  double nu, mu, dt;  // AM_VISC
  int test_m2max;     // AM_TESTF
  const double* ik2;  // 1 / |k|^2 per stored mode
  const double *visc_x, *visc_y;  // AM_VISC, FP64 handles: exp(-nu kx^2 dt), exp(-nu ky^2 dt) (NULL: computed)
  double visc_mu;
};
enum AdjKind : int { AK_NONE = 0, AK_SMAG = 1, AK_LEITH = 2 };
enum AdjProdMode : int { AP_FORWARD = 0, AP_ADJOINT = 1 };
// Pointwise products (physical arrays, working precision).
//   forward: out0 = u w_x + v w_y, out1 = g w_x, out2 = g w_y
//   adjoint: out0..3 = lam w_x, lam w_y, lam u, lam v; with a closure, p = -lam_x, q = -lam_y,
//            s = p w_x + q w_y: Leith out4,5 = g p + s w_x / g, g q + s w_y / g;
//            Smagorinsky out4,5 = g p, g q, out6,7 = 4 s psi_xy / g, s psi_d / g
struct AdjProducts {
  int kind, mode;
  const void *u, *v, *wx, *wy, *pxy, *pd;
  const void *lam, *lx, *ly;
  void* out[8];
};
constexpr int kAdjDotBlocks = 256;
// FP64 inner products, deterministic and in one launch: every block stores its partial sum, and the block that
// counts itself in last (an atomic counter, which it resets to zero) sums the partials in a fixed order.
struct AdjDotOut {
  double* partials;   // kAdjDotBlocks doubles
  double* partials2;  // kAdjDotBlocks more: the Germano pair's second sum
  unsigned* counter;  // zero between launches
  double scale;
  double* out;        // out[0] = scale * sum
  // then, if kappa is set: kappa[0] = out[0] / (n2 mm[0]) if C[0] > 0 and mm[0] > 0, else 0
  // (C_bar / (N^2 <MM>), the dynamic coefficient's share of a stage's transpose, Eq. 12, 14)
  const double* C;
  const double* mm;
  double* kappa;
  double n2;
};

template <typename T>
cudaError_t launch_adj_combine(const Geom& g, const AdjCombine& a, cudaStream_t st);
template <typename T>
cudaError_t launch_adj_products(size_t count, const AdjProducts& a, cudaStream_t st);
template <typename T>
cudaError_t launch_adj_scale(size_t count, const void* f, const void* x0, double s0, void* out0, const void* x1,
                             double s1, void* out1, cudaStream_t st);
// o.out[0] = o.scale * sum_k w_k Re(A conj B) over the stored band (w = 1 on the k_x = 0 column, else 2)
template <typename T>
cudaError_t launch_adj_spec_dot(const Geom& g, const void* A, const void* B, const AdjDotOut& o, cudaStream_t st);
// o.out[0] = o.scale * sum_i X_i Y_i Z_i
template <typename T>
cudaError_t launch_adj_phys_dot(size_t count, const void* X, const void* Y, const void* Z, const AdjDotOut& o,
                                cudaStream_t st);
// A stage's Germano sums in one pass over H and M (Eq. 12, 14): o.out[0] = o.scale <H M>, o.out[1] = o.scale
// <M M> (spectral, weighted as above), o.out[2] = C = max(0, out[0] / out[1]) if out[1] > 0, else 0
template <typename T>
cudaError_t launch_adj_germano_dots(const Geom& g, const void* H, const void* M, const AdjDotOut& o,
                                    cudaStream_t st);

// Failure-handling test: a bounded wait that runs out and sets the status flag.
cudaError_t launch_stall(int* err, cudaStream_t st);

// Sets the thread-local message returned by qg_last_error().
void set_last_error(const char* msg);

// Element-wise precision conversion between device buffers.
cudaError_t launch_convert(const void* src, int src_fp32, void* dst, int dst_fp32, size_t count, cudaStream_t st);

}  // namespace qg
