// Register-resident mixed-radix FFTs for any grid N = 2^a 3^b at run time, and the small DFTs they share with the
// compile-time engines of fast.cuh.
//
// A length-N sequence is owned by a group of TT = N / EL threads; thread t holds the EL elements at natural
// positions t + TT m.  EL is 4, 8 or 16 (N = 2^a), 12 or 18 (N with factors 3).  Every radix of the plan divides EL,
// so a Stockham pass of radix R and span NS takes EL / R butterflies per thread, butterfly j = t + TT b reading
// elements j + (N / R) r, which are the thread's own; outputs go to (j / NS) NS R + (j mod NS) + NS r through a
// padded shared-memory buffer, except in the last pass, which lands on natural ownership again.  So loads, products
// and spectral work happen in registers on the thread's own positions, and an exchange costs one barrier (two
// buffers in turn) instead of the two per pass, the integer divisions and the strided twiddle gathers of a
// transform that lives in shared memory.  The plan (radices, spans, reciprocals for the divisions, twiddle offsets)
// comes from the host; one compiled kernel per EL serves every grid of its family (RtShape).  With N known at compile
// time the same transform has every index folded (StShape, and fast.cuh): FP32 grids from 64 on have passes of their
// own, since there the integer work of a run-time length is most of the instructions (Smagorinsky 1296^2: 1296 us per
// step with the shared-memory transforms, 666 with the run-time ones, 298 with passes for N = 1296).
//
// Only the forward kernel exp(-2 pi i / N) is compiled: an inverse transform is the forward one of the sequence
// with real and imaginary parts exchanged, its result exchanged again, which costs nothing where the parts are
// loaded and stored one by one.
#pragma once

#include <vector>

#include "qg_common.cuh"

namespace qg {

// Radices of a length-n transform with el elements per thread: the largest allowed ones first, which also gives the
// fewest passes for every n = 2^a 3^b up to 4096.
constexpr int kMaxPass = 8;
struct Radices {
  int np;  // number of passes, 0 if n has no such factorisation
  int radix[kMaxPass], ns[kMaxPass], off[kMaxPass];
  int table;
};
constexpr Radices fft_radices(int n, int el) {
  const int sets[5][5] = {{4, 2, 0, 0, 0}, {8, 4, 2, 0, 0}, {16, 8, 4, 2, 0}, {12, 6, 4, 3, 2}, {18, 9, 6, 3, 2}};
  const int s = el == 4 ? 0 : el == 8 ? 1 : el == 16 ? 2 : el == 12 ? 3 : 4;
  Radices r{};
  if (n % el) return r;
  int m = n, ns = 1, off = 0;
  while (m > 1) {
    int R = 0;
    for (int i = 0; i < 5 && !R; ++i)
      if (sets[s][i] && m % sets[s][i] == 0) R = sets[s][i];
    if (!R || r.np == kMaxPass) return Radices{};
    r.radix[r.np] = R;
    r.ns[r.np] = ns;
    r.off[r.np] = off;
    if (ns > 1) off += (R - 1) * ns;
    ns *= R;
    m /= R;
    ++r.np;
  }
  r.table = off > 0 ? off : 1;
  return r;
}
// Elements per thread of the FP32 passes specialised for n: eight up to 512 (a grid with few rows has idle SMs, and
// half as many elements per thread halve the chain), sixteen above (one exchange fewer).  Factors of 3, in any pass:
// twelve or eighteen, whichever needs fewer passes.
constexpr int fft_elems(int n) {
  if (n % 3) return n <= 512 ? 8 : 16;
  const int a = fft_radices(n, 12).np, b = fft_radices(n, 18).np;
  return a && (!b || a <= b) ? 12 : 18;
}

// The same for the run-time passes.  FP64, n = 2^a: four -- on this GPU an FP64 instruction occupies its quarter of an
// SM for 64 cycles at best (spectral.cuh), so a transform's time is its FP64 operations, spread over as many warps as possible; eight
// at 4096, where four would take more threads than a CTA has.  A 2^a grid of FP32 reals keeps eight (its larger grids
// have passes of their own).
constexpr int rt_elems(int n, int esz) { return n % 3 ? (esz == 8 && n <= 2048 ? 4 : 8) : fft_elems(n); }
// most threads of a CTA of the run-time passes: twelve and eighteen FP64 elements need 168 registers a thread
constexpr int pass_threads(int el, int esz) { return esz == 8 && el > 8 ? 384 : 512; }

struct FftPass {
  int radix;
  int ns;        // span: the product of the earlier radices
  unsigned inv;  // floor(2^32 / ns) + 1: j / ns = umulhi(j, inv) for j < 4096 (unused for ns = 1)
  int off;       // this pass's twiddles: [r - 1][k], k < ns, at off + (r - 1) ns + k
};
struct FftPlan {
  int n = 0;
  int el = 0, tt = 0;  // elements per thread, threads per sequence
  int npass = 0;
  int buf = 0;         // complex elements of one padded exchange buffer
  int table = 0;       // complex entries of the twiddle table
  FftPass pass[kMaxPass] = {};
};

// plan for n = 2^a 3^b (even, 16..4096) with el elements per thread
FftPlan fft_plan(int n, int el);
// Entry e of the plan's twiddle table belongs to a pass of this radix and stands for w = exp(-2 pi i j / n) with this
// j = r k n / (ns R).
struct FftEntry {
  int j, radix;
};
__host__ __device__ inline FftEntry fft_table_entry(const FftPlan& p, int e) {
  for (int i = p.npass - 1; i >= 1; --i) {
    const FftPass& s = p.pass[i];
    if (e < s.off) continue;
    const int r = (e - s.off) / s.ns + 1, k = (e - s.off) % s.ns;
    return {(int)(((long long)r * k * (p.n / (s.ns * s.radix))) % p.n), s.radix};
  }
  return {0, 0};
}
// FP64 passes of radix 2 and 4 take a twiddle w = c + i s as (c, s / c) (see twiddled), others as (c, s)
__host__ __device__ constexpr bool ratio_twiddle(int radix, int esz) { return esz == 8 && (radix == 2 || radix == 4); }
// for w = +-i, c is this instead of 0: c (s / c) is s still, and c itself, 1e-18, is nothing beside it
constexpr double kRatioMinCos = 1.0 / (1ll << 60);
// the table of the plan for elements of esz bytes (plan.cu): pairs of doubles, each the rounding of its exact value
std::vector<double> fft_table(const FftPlan& p, int esz);

template <typename C> __device__ __forceinline__ C cmulk(C a, decltype(C::x) c, decltype(C::x) s) {
  return mk<C>(a.x * c - a.y * s, a.x * s + a.y * c);
}

// Complex sums and differences of the butterflies.  With QG_PACKED_F32 (the default) the FP32 forms use the
// packed pair instructions of the sm_100 family (add / sub .rn.f32x2): both parts in one instruction, each part
// rounded as the scalar operation rounds it.  The transforms then issue 14% fewer instructions; results differ
// from the scalar build only where the compiler had fused one of these sums into a neighbouring product (an FMA,
// one rounding fewer), at the level of FP32 rounding.
#ifndef QG_PACKED_F32
#define QG_PACKED_F32 1
#endif
__device__ __forceinline__ unsigned long long f2_bits(float2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ float2 bits_f2(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
template <typename C, bool PK> __device__ __forceinline__ C vadd(C a, C b) {
  if constexpr (QG_PACKED_F32 && PK && std::is_same<C, float2>::value) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return bits_f2(r);
  } else {
    return cadd(a, b);
  }
}
template <typename C, bool PK> __device__ __forceinline__ C vsub(C a, C b) {
  if constexpr (QG_PACKED_F32 && PK && std::is_same<C, float2>::value) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return bits_f2(r);
  } else {
    return csub(a, b);
  }
}
// a b + c, part by part (one instruction, each part rounded as fmaf rounds it)
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)), "l"(f2_bits(c)));
  return bits_f2(r);
}
// plus = t + i s d, minus = t - i s d (s = +1 / -1) with the parts of d exchanged in place
template <typename C> __device__ __forceinline__ void rot_pm(C t, C d, int s, C& plus, C& minus) {
  if (s > 0) {
    plus = mk<C>(t.x - d.y, t.y + d.x);
    minus = mk<C>(t.x + d.y, t.y - d.x);
  } else {
    plus = mk<C>(t.x + d.y, t.y - d.x);
    minus = mk<C>(t.x - d.y, t.y + d.x);
  }
}

// 4-, 8- and 2-point DFTs with kernel exp(s 2 pi i n k / R)
template <typename C, bool PK> __device__ __forceinline__ void dft4v(C* v, int s) {
  const C t0 = vadd<C, PK>(v[0], v[2]);
  const C t1 = vsub<C, PK>(v[0], v[2]);
  const C t2 = vadd<C, PK>(v[1], v[3]);
  const C d = vsub<C, PK>(v[1], v[3]);
  v[0] = vadd<C, PK>(t0, t2);
  v[2] = vsub<C, PK>(t0, t2);
  rot_pm(t1, d, s, v[1], v[3]);
}
template <typename C, bool PK> __device__ __forceinline__ void dft8v(C* v, int s) {
  using T = decltype(C::x);
  const T h = T(0.70710678118654752440);
  C e[4] = {v[0], v[2], v[4], v[6]};
  C o[4] = {v[1], v[3], v[5], v[7]};
  dft4v<C, PK>(e, s);
  dft4v<C, PK>(o, s);
  // o[m] *= w8^m, w8 = exp(s 2 pi i / 8) = (1 + s i) / sqrt 2
  const C o1 = mk<C>((o[1].x - s * o[1].y) * h, (o[1].y + s * o[1].x) * h);
  const C o3 = mk<C>((-o[3].x - s * o[3].y) * h, (-o[3].y + s * o[3].x) * h);
  v[0] = vadd<C, PK>(e[0], o[0]);
  v[4] = vsub<C, PK>(e[0], o[0]);
  v[1] = vadd<C, PK>(e[1], o1);
  v[5] = vsub<C, PK>(e[1], o1);
  rot_pm(e[2], o[2], s, v[2], v[6]);
  v[3] = vadd<C, PK>(e[3], o3);
  v[7] = vsub<C, PK>(e[3], o3);
}
template <typename C, bool PK> __device__ __forceinline__ void dft2v(C* v) {
  const C a = v[0], b = v[1];
  v[0] = vadd<C, PK>(a, b);
  v[1] = vsub<C, PK>(a, b);
}

template <typename C, bool PK> __device__ __forceinline__ void dft16(C* v, int s) {
  using T = decltype(C::x);
  const T c1 = T(0.92387953251128675613);  // cos(pi/8)
  const T s1 = T(0.38268343236508977173);  // sin(pi/8)
  const T h = T(0.70710678118654752440);
  C a[4][4];
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) {
    C q[4] = {v[n2], v[4 + n2], v[8 + n2], v[12 + n2]};
    dft4v<C, PK>(q, s);
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) a[n2][k1] = q[k1];
  }
  // a[n2][k1] *= exp(s 2 pi i n2 k1 / 16)
  const T ss = T(s);
  a[1][1] = cmulk(a[1][1], c1, ss * s1);
  a[1][2] = cmulk(a[1][2], h, ss * h);
  a[1][3] = cmulk(a[1][3], s1, ss * c1);
  a[2][1] = cmulk(a[2][1], h, ss * h);
  a[2][2] = cmul_si(a[2][2], s);
  a[2][3] = cmulk(a[2][3], -h, ss * h);
  a[3][1] = cmulk(a[3][1], s1, ss * c1);
  a[3][2] = cmulk(a[3][2], -h, ss * h);
  a[3][3] = cmulk(a[3][3], -c1, -ss * s1);
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
    C q[4] = {a[0][k1], a[1][k1], a[2][k1], a[3][k1]};
    dft4v<C, PK>(q, s);
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = q[k2];
  }
}

// 3-point DFT with kernel exp(s 2 pi i n k / 3)
template <typename C, bool PK> __device__ __forceinline__ void dft3(C* v, int s) {
  using T = decltype(C::x);
  const T h = T(0.86602540378443864676);  // sin(pi/3)
  const C a = v[0];
  const C bc = vadd<C, PK>(v[1], v[2]);
  const C d = vsub<C, PK>(v[1], v[2]);
  const C m = mk<C>(a.x - T(0.5) * bc.x, a.y - T(0.5) * bc.y);
  v[0] = vadd<C, PK>(a, bc);
  // m +- i s sin(pi/3) (v1 - v2).  FP64: the rounded sine is 5.8e-17 too small, which would shrink every transform's
  // result a little, step after step; the second output takes the next number above, 7.0e-17 too large
  // (12 steps at 162^2 end 8.8e-15 from an 80-bit run with the one constant and 6.4e-15 with the two).
  if constexpr (sizeof(T) == 8) {
    const T up = T(0.86602540378443870761);
    C other;
    rot_pm(m, cscale(d, h), s, v[1], other);
    rot_pm(m, cscale(d, up), s, other, v[2]);
  } else {
    rot_pm(m, cscale(d, h), s, v[1], v[2]);
  }
}

// The 6-, 12- and 18-point DFTs take their coprime factors by the prime-factor index maps (Good, 1958; Thomas, 1963:
// n by multiples, k by the Chinese remainder theorem), which leave no factor between the two stages.  The twiddle
// products of the mixed-radix form cost operations, and their rounded constants (sin 60 degrees above all, off by the
// same sign in every one of them) added up from step to step: 20 FP64 steps at 72^2 ended 1.5e-14 from an 80-bit run,
// with these forms 6.8e-15, in 5.68 ms against 6.05 (648^2, four steps: 4.4e-15 and 3.5e-15, 6.38 and 5.86 ms).

// 12-point DFT: n = 4 n1 + 3 n2, k = 4 k1 + 9 k2 (mod 12), 4-point DFTs over n2, 3-point DFTs over n1
template <typename C, bool PK> __device__ __forceinline__ void dft12(C* v, int s) {
  C a[3][4];
#pragma unroll
  for (int n1 = 0; n1 < 3; ++n1) {
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) a[n1][n2] = v[(4 * n1 + 3 * n2) % 12];
    dft4v<C, PK>(a[n1], s);
  }
#pragma unroll
  for (int k2 = 0; k2 < 4; ++k2) {
    C q[3] = {a[0][k2], a[1][k2], a[2][k2]};
    dft3<C, PK>(q, s);
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) v[(4 * k1 + 9 * k2) % 12] = q[k1];
  }
}

// 6-point DFT: n = 3 n1 + 2 n2, k = 3 k1 + 4 k2 (mod 6), 3-point DFTs over n2, sums and differences over n1
template <typename C, bool PK> __device__ __forceinline__ void dft6(C* v, int s) {
  C e[3] = {v[0], v[2], v[4]}, o[3] = {v[3], v[5], v[1]};
  dft3<C, PK>(e, s);
  dft3<C, PK>(o, s);
#pragma unroll
  for (int k2 = 0; k2 < 3; ++k2) {
    v[(4 * k2) % 6] = vadd<C, PK>(e[k2], o[k2]);
    v[(3 + 4 * k2) % 6] = vsub<C, PK>(e[k2], o[k2]);
  }
}

// 9-point DFT as 3 x 3: n = 3 n1 + n2, k = k1 + 3 k2, twiddles exp(s 2 pi i n2 k1 / 9)
template <typename C, bool PK> __device__ __forceinline__ void dft9(C* v, int s) {
  using T = decltype(C::x);
  const T ss = T(s);
  const T c1 = T(0.76604444311897803520), s1 = T(0.64278760968653932632);   // 40 degrees
  const T c2 = T(0.17364817766693034885), s2 = T(0.98480775301220805937);   // 80
  const T c4 = T(-0.93969262078590838405), s4 = T(0.34202014332566873304);  // 160
  C a[3][3];
#pragma unroll
  for (int n2 = 0; n2 < 3; ++n2) {
    C q[3] = {v[n2], v[3 + n2], v[6 + n2]};
    dft3<C, PK>(q, s);
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) a[n2][k1] = q[k1];
  }
  a[1][1] = cmulk(a[1][1], c1, ss * s1);
  a[1][2] = cmulk(a[1][2], c2, ss * s2);
  a[2][1] = cmulk(a[2][1], c2, ss * s2);
  a[2][2] = cmulk(a[2][2], c4, ss * s4);
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) {
    C q[3] = {a[0][k1], a[1][k1], a[2][k1]};
    dft3<C, PK>(q, s);
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = q[k2];
  }
}

// 18-point DFT: n = 9 n1 + 2 n2, k = 9 k1 + 10 k2 (mod 18), 9-point DFTs over n2, sums and differences over n1
template <typename C, bool PK> __device__ __forceinline__ void dft18(C* v, int s) {
  C e[9], o[9];
#pragma unroll
  for (int n2 = 0; n2 < 9; ++n2) {
    e[n2] = v[2 * n2];
    o[n2] = v[(9 + 2 * n2) % 18];
  }
  dft9<C, PK>(e, s);
  dft9<C, PK>(o, s);
#pragma unroll
  for (int k2 = 0; k2 < 9; ++k2) {
    v[(10 * k2) % 18] = vadd<C, PK>(e[k2], o[k2]);
    v[(9 + 10 * k2) % 18] = vsub<C, PK>(e[k2], o[k2]);
  }
}

template <typename C, int R, bool PK> __device__ __forceinline__ void dftR(C* v, int s) {
  if constexpr (R == 18) dft18<C, PK>(v, s);
  else if constexpr (R == 16) dft16<C, PK>(v, s);
  else if constexpr (R == 12) dft12<C, PK>(v, s);
  else if constexpr (R == 9) dft9<C, PK>(v, s);
  else if constexpr (R == 8) dft8v<C, PK>(v, s);
  else if constexpr (R == 6) dft6<C, PK>(v, s);
  else if constexpr (R == 4) dft4v<C, PK>(v, s);
  else if constexpr (R == 3) dft3<C, PK>(v, s);
  else dft2v<C, PK>(v);
}

// one shared-memory padding element every 16
__host__ __device__ __forceinline__ int fft_pad(int i) { return i + (i >> 4); }

// The exchange buffers of one sequence and their barrier.  Groups that lie inside a warp exchange under a warp
// barrier, others under the CTA's (then every thread of the CTA runs the same passes).
template <typename C> struct FftBufs {
  C* b[2];      // equal when the CTA has one buffer per sequence (a second barrier then guards its reuse)
  int ph = 0;   // buffer of the next exchange
  bool one;     // b[0] == b[1]
  bool warp;    // the group lies inside a warp
  bool active;  // this thread belongs to a group (the others only take part in the barriers)
  int* st;      // status bits of the bounds-checked debug build
  int len;      // elements of a buffer
  __device__ __forceinline__ void sync() const {
    if (warp) __syncwarp();
    else __syncthreads();
  }
  // the buffer every thread of the group has finished reading; with one buffer after a barrier
  __device__ __forceinline__ C* take() {
    if (one) sync();
    C* r = b[ph];
    ph ^= 1;
    return r;
  }
};

// b (1 + i q) = b w / c for the twiddle w = c (1 + i q), given as (c, q)
template <typename C> __device__ __forceinline__ C tw_turn(C b, C w) {
  return mk<C>(fma(-w.y, b.y, b.x), fma(w.y, b.x, b.y));
}
// (a, b) <- (a + c b, a - c b)
template <typename C> __device__ __forceinline__ void tw_sums(C& a, C& b, decltype(C::x) c) {
  const C s = mk<C>(fma(c, b.x, a.x), fma(c, b.y, a.y));
  b = mk<C>(fma(-c, b.x, a.x), fma(-c, b.y, a.y));
  a = s;
}
// Butterfly of radix R with its twiddles w[(r - 1) ns] (kernel exp(s 2 pi i / N): conjugated for s > 0).  FP64 radices
// 2 and 4 take them as cosine and tangent, the cosine joining the first sums (Linzer and Feig, "Implementation of
// efficient FFT algorithms on fused multiply-add architectures", 1993): six operations for radix 2 against eight, 24
// for radix 4 against 28.  Every element meets one table entry and every sum rounds once.  Forming a difference as
// 2 a minus the sum, and v3's twiddle as a product of two entries, takes 24 operations too, but adds the sum's and
// the second entry's roundings.
// GL: the table lies in global memory (else in shared memory or anywhere).
template <bool GL, typename C> __device__ __forceinline__ C tw_load(const C* w) {
  if constexpr (GL) return __ldg(w);
  else return *w;
}
template <typename C, int R, bool PK, bool GL>
__device__ __forceinline__ void twiddled(C* v, const C* w, int ns, int s) {
  using T = decltype(C::x);
  if constexpr (ratio_twiddle(R, sizeof(T))) {
    C w1 = tw_load<GL>(w);
    if (s > 0) w1.y = -w1.y;
    v[1] = tw_turn(v[1], w1);
    if constexpr (R == 2) {
      tw_sums(v[0], v[1], w1.x);
    } else {
      C w2 = tw_load<GL>(w + ns), w3 = tw_load<GL>(w + 2 * ns);
      if (s > 0) {
        w2.y = -w2.y;
        w3.y = -w3.y;
      }
      C a = v[0], b = tw_turn(v[2], w2), c = cscale(v[1], w1.x), d = tw_turn(v[3], w3);
      tw_sums(a, b, w2.x);
      tw_sums(c, d, w3.x);
      v[0] = cadd(a, c);
      v[2] = csub(a, c);
      rot_pm(b, d, s, v[1], v[3]);
    }
  } else {
#pragma unroll
    for (int r = 1; r < R; ++r) {
      C wr = tw_load<GL>(w + (r - 1) * ns);
      if (s > 0) wr.y = -wr.y;
      v[r] = cmul(v[r], wr);
    }
    dftR<C, R, PK>(v, s);
  }
}

// The twiddle table of a small plan moves to shared memory at the start of a pass: read from L2 by every pass of
// every transform it would be most of a short transform's latency.  Larger tables stay in global memory (L1).
constexpr int kTwShared = 512;  // entries
__host__ __device__ constexpr bool tw_shared(int table) { return table <= kTwShared; }
template <typename C> __device__ __forceinline__ const C* tw_stage(const C* tw, int table, C* sm) {
  if (!tw_shared(table)) return tw;
  for (int i = threadIdx.x; i < table; i += blockDim.x) sm[i] = __ldg(tw + i);
  return sm;  // complete at the next CTA barrier
}

// The run-time transform: EL elements per thread, the plan in a kernel parameter.
template <int EL_> struct RtShape {
  static constexpr int EL = EL_;
  FftPlan p;
  __device__ __forceinline__ int n() const { return p.n; }
  __device__ __forceinline__ int tt() const { return p.tt; }
  __device__ __forceinline__ int buf() const { return p.buf; }
  __device__ __forceinline__ int table() const { return p.table; }
  __device__ __forceinline__ int band(const Geom& g) const { return g.K; }

  template <int R, typename C>
  __device__ __forceinline__ void pass(C* x, int t, const FftPass& ps, bool last, C* buf, const C* tw,
                                       const FftBufs<C>& fb) const {
    constexpr int NB = EL / R;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int j = t + p.tt * b;
      C v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = x[b + NB * r];
      int q = j, k = 0;
      if (ps.ns > 1) {
        q = __umulhi((unsigned)j, ps.inv);
        k = j - q * ps.ns;
        twiddled<C, R, true, false>(v, tw + ps.off + k, ps.ns, -1);
      } else {
        dftR<C, R, true>(v, -1);
      }
      if (last) {
#pragma unroll
        for (int r = 0; r < R; ++r) x[b + NB * r] = v[r];
      } else {
        const int base = q * ps.ns * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) QG_ST(buf, fft_pad(base + ps.ns * r), fb.len, fb.st, v[r]);
      }
    }
  }

  // forward transform, natural ownership in and out
  template <typename C>
  __device__ __forceinline__ void run(C* x, int t, FftBufs<C>& fb, const C* tw) const {
#pragma unroll 1
    for (int i = 0; i < p.npass; ++i) {
      const FftPass ps = p.pass[i];
      const bool last = i == p.npass - 1;
      C* buf = last ? nullptr : fb.take();
      if (fb.active) switch (ps.radix) {
        case 2: pass<2>(x, t, ps, last, buf, tw, fb); break;
        case 3: if constexpr (EL % 3 == 0) pass<3>(x, t, ps, last, buf, tw, fb); break;
        case 4: if constexpr (EL % 4 == 0) pass<4>(x, t, ps, last, buf, tw, fb); break;
        case 6: if constexpr (EL % 6 == 0) pass<6>(x, t, ps, last, buf, tw, fb); break;
        case 8: if constexpr (EL % 8 == 0) pass<8>(x, t, ps, last, buf, tw, fb); break;
        case 9: if constexpr (EL % 9 == 0) pass<9>(x, t, ps, last, buf, tw, fb); break;
        case 12: if constexpr (EL % 12 == 0) pass<12>(x, t, ps, last, buf, tw, fb); break;
        case 18: if constexpr (EL % 18 == 0) pass<18>(x, t, ps, last, buf, tw, fb); break;
      }
      if (!last) {
        fb.sync();
        if (fb.active) {
#pragma unroll
          for (int m = 0; m < EL; ++m) x[m] = QG_LD(buf, fft_pad(t + p.tt * m), fb.len, fb.st);
        }
      }
    }
  }
};

// Pass I of the compile-time transform of length N: x in natural ownership on entry; a non-last pass writes its
// outputs to buf (when active; len elements, status bits st in the bounds-checked debug build), the last one leaves
// them in x.
template <typename C, int N, int EL, int I, bool PK, bool GL>
__device__ __forceinline__ void st_pass(C* x, int t, C* buf, const C* tw, int s, bool active, int len, int* st) {
  (void)len; (void)st;
  constexpr Radices P = fft_radices(N, EL);
  constexpr int R = P.radix[I], NS = P.ns[I], NB = EL / R, TT = N / EL;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int j = t + TT * b;
    const int k = j % NS;
    C v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = x[b + NB * r];
    if constexpr (NS > 1) twiddled<C, R, PK, GL>(v, tw + P.off[I] + k, NS, s);
    else dftR<C, R, PK>(v, s);
    if constexpr (I == P.np - 1) {
#pragma unroll
      for (int r = 0; r < R; ++r) x[b + NB * r] = v[r];
    } else if (active) {
      const int base = (j / NS) * NS * R + k;
#pragma unroll
      for (int r = 0; r < R; ++r) QG_ST(buf, fft_pad(base + NS * r), len, st, v[r]);
    }
  }
}

// The compile-time transform: the same plan and interface, every index a constant expression of the thread.
template <int N_, int EL_> struct StShape {
  static constexpr int EL = EL_;
  __device__ __forceinline__ constexpr int n() const { return N_; }
  __device__ __forceinline__ constexpr int tt() const { return N_ / EL_; }
  __device__ __forceinline__ constexpr int buf() const { return N_ + N_ / 16 + 1; }
  __device__ __forceinline__ constexpr int table() const { return fft_radices(N_, EL_).table; }
  __device__ __forceinline__ constexpr int band(const Geom&) const { return (N_ - 1) / 3; }

  template <int I, typename C>
  __device__ __forceinline__ void from(C* x, int t, FftBufs<C>& fb, const C* tw) const {
    constexpr int np = fft_radices(N_, EL_).np;
    if constexpr (I < np) {
      constexpr bool last = I == np - 1;
      C* buf = last ? nullptr : fb.take();
      st_pass<C, N_, EL_, I, true, false>(x, t, buf, tw, -1, fb.active, fb.len, fb.st);
      if constexpr (!last) {
        fb.sync();
#pragma unroll
        for (int m = 0; m < EL; ++m) x[m] = QG_LD(buf, fft_pad(t + N_ / EL_ * m), fb.len, fb.st);
        from<I + 1>(x, t, fb, tw);
      }
    }
  }
  template <typename C>
  __device__ __forceinline__ void run(C* x, int t, FftBufs<C>& fb, const C* tw) const {
    from<0>(x, t, fb, tw);
  }
};

}  // namespace qg
