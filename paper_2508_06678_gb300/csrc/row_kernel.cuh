// Row pass: for physical rows y, inverse x-transform every incoming field, form the pointwise products of the step
// in physical space (collocation, Sec. II-C), and forward x-transform the products.
//
// Two real rows share one complex N-point FFT: inputs are packed as Z = A + i B with the Hermitian extension of the
// two half spectra, outputs are split with A = (Z_k + conj Z_{N-k}) / 2, B = (Z_k - conj Z_{N-k}) / 2i.  Only the
// kept columns m_x <= K are read or written (2/3 rule).
//
// Products (per grid point, working precision):
//   J  = u_total w_x + v w_y                             (Eq. 1)
//   g  = |grad w| = sqrt(w_x^2 + w_y^2)                  (Eq. 13)
//   g  = |S| = sqrt(4 psi_xy^2 + (psi_xx - psi_yy)^2)    (Eq. 10)
//   P  = g w_x (times i k_x after the transform),  Q = g w_y   (Eq. 9)
//   Brinkman / sponge: f <- f * exp(-rate chi dt)        (Eq. 2, 3; exact)
#pragma once

#include "fft.cuh"
#include "qg_kernels.h"

namespace qg {

// Task i of a pass over `rows` rows with nf fields per row: the two (row, field) items that share one complex
// transform; the odd field of a row pairs with the next row's (rb = -1: no second item).
struct RowTask {
  int ra, fa, rb, fb;
};
__device__ __forceinline__ int row_tasks(int rows, int nf) { return rows * (nf / 2) + (nf & 1 ? (rows + 1) / 2 : 0); }
__device__ __forceinline__ RowTask row_task(int i, int rows, int nf) {
  const int half = nf / 2;
  RowTask k;
  if (i < rows * half) {
    k.ra = k.rb = i / half;
    k.fa = 2 * (i - k.ra * half);
    k.fb = k.fa + 1;
  } else {
    const int l = 2 * (i - rows * half);
    k.ra = l;
    k.fa = k.fb = nf - 1;
    k.rb = l + 1 < rows ? l + 1 : -1;
  }
  return k;
}

template <typename T> struct PtProducts {
  static __device__ __forceinline__ void leith(T u, T v, T wx, T wy, T& J, T& P, T& Q) {
    J = u * wx + v * wy;
    const T g = sqrt(wx * wx + wy * wy);
    P = g * wx;
    Q = g * wy;
  }
  static __device__ __forceinline__ void smag(T u, T v, T wx, T wy, T pxy, T pd, T& J, T& P, T& Q) {
    J = u * wx + v * wy;
    const T g = sqrt(T(4) * pxy * pxy + pd * pd);
    P = g * wx;
    Q = g * wy;
  }
};

// One CTA takes c.rows rows with c.groups groups of TT threads, each transforming one pair of real rows at a time.
// The physical rows meet in shared memory (slots) for the products, so the transforms of a row run side by side:
// a small grid has too few rows to fill the chip with one row per group, and its passes are as long as one row's
// chain of transforms.  Programs that only scale or copy keep their pair in registers and use no slots.
// FP64 (every grid) is bound by its FP64 operations: what counts is that all SMs have them and that there are few, so
// conversions, divisions and finiteness tests go through tables and integer operations.  Measured per step, against
// the shared-memory transforms these passes replaced (or, FP64 from 256 on and FP32 256, the passes that run a row's
// transforms one after another with sixteen elements per thread): FP64 Smagorinsky 128^2 463 -> 144 us, FP64 no
// closure 1024^2 2101 -> 1533 us, FP32 dynamic Smagorinsky 256^2 152 -> 92 us.
template <typename T, class Sh, int PROG>
__global__ void __launch_bounds__(pass_threads(Sh::EL, sizeof(T))) row_kernel(Geom g, Sh sh, RowConfig c, RowDesc d,
                                                                 const cplx_t<T>* __restrict__ twg) {
  using C = cplx_t<T>;
  constexpr int EL = Sh::EL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = sh.n(), K = sh.band(g);
  const int tid = threadIdx.x, nt = blockDim.x;
  const int gi = tid / sh.tt(), t = tid - gi * sh.tt();
  const int rows = (int)blockIdx.x < c.full ? c.rows : 1;
  const int y0 = (int)blockIdx.x < c.full ? blockIdx.x * c.rows : c.full * c.rows + (blockIdx.x - c.full);
  int* const st = d.err;
  // extents for the bounds-checked debug build
  const long long n_mixed = (long long)N * g.IP, n_phys = (long long)N * N;
  C* const tws = reinterpret_cast<C*>(smem_raw);
  C* const bufs = tws + (tw_shared(sh.table()) ? sh.table() : 0);
  const C* tw = tw_stage(twg, sh.table(), tws);
  pdl_enter();
  const int stop = d.flag ? *reinterpret_cast<volatile int*>(d.flag) : 0;
  T* const slots = reinterpret_cast<T*>(bufs + (size_t)c.groups * (c.one_buf ? 1 : 2) * sh.buf());
  const long long nslot_el = (long long)c.rows * c.nslot * N;
  (void)n_mixed; (void)n_phys; (void)nslot_el; (void)st;
  FftBufs<C> fb;
  fb.active = gi < c.groups;
  fb.one = c.one_buf;
  fb.warp = c.warp;
  fb.st = st;
  fb.len = sh.buf();
  fb.b[0] = bufs + (size_t)(fb.active ? gi : 0) * (c.one_buf ? 1 : 2) * sh.buf();
  fb.b[1] = c.one_buf ? fb.b[0] : fb.b[0] + sh.buf();

  constexpr bool direct = PROG == RP_SCALE || PROG == RP_COPY;
  constexpr bool smag4 = PROG == RP_SMAG || PROG == RP_DSMAG;
  // direct programs transform item pairs that never meet: field f of row r in, the same item out
  const int nitem = direct ? (d.npair > 0 ? 2 * d.npair : d.in_phys ? d.nout : d.nin) : d.nin;
  const int tin = row_tasks(rows, nitem);
  const int tout = direct ? tin : row_tasks(rows, d.nout);
  const bool has_inv = PROG != RP_COPY || !d.in_phys, has_fwd = PROG == RP_SCALE || d.in_phys;  // of a direct program
  int bad = 0;
  C x[EL];
#pragma unroll
  for (int m = 0; m < EL; ++m) x[m] = mk<C>(T(0), T(0));

  // packed pair (a, b)(k) of mixed rows as the transform's input at element k, parts exchanged (inverse)
  auto load_pair = [&](auto pair) {
#pragma unroll
    for (int m = 0; m < EL; ++m) {
      const int k = t + sh.tt() * m;
      C z = mk<C>(T(0), T(0));
      if (k <= K || k >= N - K) {
        const int kk = k <= K ? k : N - k;
        C a, b;
        pair(kk, a, b);
        if (k == 0) {
          a.y = T(0);
          b.y = T(0);
        }
        z = k <= K ? mk<C>(a.x - b.y, a.y + b.x) : mk<C>(a.x + b.y, b.x - a.y);
      }
      x[m] = mk<C>(z.y, z.x);
    }
  };

  // rounds: inverse tasks (to the slots), then forward tasks; direct programs alternate per task
  const int rin = (tin + c.groups - 1) / c.groups, rout = (tout + c.groups - 1) / c.groups;
  const int nround = direct ? rin * ((has_inv ? 1 : 0) + (has_fwd ? 1 : 0)) : rin + rout;
#pragma unroll 1
  for (int it = 0; it < nround; ++it) {
    bool inv;
    int base;
    if (!direct) {
      inv = it < rin;
      base = (inv ? it : it - rin) * c.groups;
    } else if (has_inv && has_fwd) {
      inv = !(it & 1);
      base = (it >> 1) * c.groups;
    } else {
      inv = has_inv;
      base = it * c.groups;
    }
    const int task = base + gi;
    const bool on = fb.active && task < (inv ? tin : tout);
    RowTask k2 = {0, 0, -1, 0};
    if (on) k2 = row_task(task, rows, (inv || direct) ? nitem : d.nout);
    const int ya = y0 + k2.ra, yb = y0 + (k2.rb >= 0 ? k2.rb : 0);
    // an absent second field of a copy pair
    const bool two = on && k2.rb >= 0 && !(d.npair > 0 && (d.in_phys ? d.pin[k2.fb] : d.pout[k2.fb]) == nullptr);

    // ---- the transform's input
    if (on) {
      if (inv) {
        const int oa = ya * g.IP, ob = yb * g.IP;
        (void)ob;
        auto ld = [&](int i, int at) { return QG_LD(reinterpret_cast<const C*>(d.in[i]), at, n_mixed, st); };
        if constexpr (smag4) {
          // The Smagorinsky programs read u, v, w, w_y of a level: in mixed space (k_x, y) the derivatives in x are
          // factors, so w_x = i k_x w and, with u = -psi_y + U, v = psi_x and psi_yy = w - psi_xx, the strain pair
          // is psi_xy = -i k_x u (the mean U sits at k_x = 0) and psi_xx - psi_yy = 2 i k_x v - w.
          const int l = k2.fa >= 6 ? 4 : 0, q = k2.fa - (k2.fa >= 6 ? 6 : 0);
          if (q == 0)
            load_pair([&](int k, C& a, C& b) { a = ld(l, oa + k); b = ld(l + 1, oa + k); });
          else if (q == 2)
            load_pair([&](int k, C& a, C& b) { a = cmul_ik(ld(l + 2, oa + k), wavenumber<T>(g, k)); b = ld(l + 3, oa + k); });
          else
            load_pair([&](int k, C& a, C& b) {
              const T kx = wavenumber<T>(g, k);
              a = cmul_ik(ld(l, oa + k), -kx);
              b = csub(cmul_ik(ld(l + 1, oa + k), T(2) * kx), ld(l + 2, oa + k));
            });
        } else {
          load_pair([&](int k, C& a, C& b) {
            a = ld(k2.fa, oa + k);
            b = two ? ld(k2.fb, ob + k) : mk<C>(T(0), T(0));
          });
        }
      } else if (!direct) {
        const int oa = (k2.ra * c.nslot + k2.fa) * N, ob = ((two ? k2.rb : 0) * c.nslot + k2.fb) * N;
#pragma unroll
        for (int m = 0; m < EL; ++m) {
          const int k = t + sh.tt() * m;
          x[m] = mk<C>(QG_LD(slots, oa + k, nslot_el, st), two ? QG_LD(slots, ob + k, nslot_el, st) : T(0));
        }
      } else if (d.in_phys) {
        const bool batch = d.npair > 0;
        const T* pa = reinterpret_cast<const T*>(batch ? d.pin[k2.fa] : k2.fa ? d.phys_in2 : d.phys_in);
        const T* pb = reinterpret_cast<const T*>(batch ? d.pin[k2.fb] : k2.fb ? d.phys_in2 : d.phys_in);
#pragma unroll
        for (int m = 0; m < EL; ++m) {
          const int k = t + sh.tt() * m;
          x[m] = mk<C>(QG_LD(pa, ya * N + k, n_phys, st),
                       two ? QG_LD(pb, yb * N + k, n_phys, st) : T(0));
        }
      }
    }

    // the status flag's load has overlapped the inputs'; the barrier also completes the twiddle table
    if (it == 0 && __syncthreads_or(stop)) return;
    sh.run(x, t, fb, tw);

    // ---- where the result goes
    if (inv) {
      if (!direct) {
        if (on) {
#pragma unroll
          for (int m = 0; m < EL; ++m) {
            const int k = t + sh.tt() * m;
            QG_ST(slots, (k2.ra * c.nslot + k2.fa) * N + k, nslot_el, st, x[m].y);
            if (two) QG_ST(slots, (k2.rb * c.nslot + k2.fb) * N + k, nslot_el, st, x[m].x);
          }
        }
        if (it == rin - 1) {
          __syncthreads();
          // ---- pointwise products, in place in the slots
          const int total = rows * N;
          for (int e = tid; e < total; e += nt) {
            const int r = e >= N ? 1 : 0, xx = e - r * N;  // at most two rows
            T* s = slots + (size_t)r * c.nslot * N + xx;
#ifdef QG_CHECKED
            if (!QG_INB((long long)(r + 1) * c.nslot * N - N + xx, nslot_el, st)) continue;
#endif
#define S(i) s[(size_t)(i) * N]
            const int px = (y0 + r) * N + xx;
            (void)px;
            if constexpr (PROG == RP_NONE) {
              const T J = S(0) * S(2) + S(1) * S(3);
              S(0) = J;
            } else if constexpr (PROG == RP_LEITH) {
              T J, P, Q;
              PtProducts<T>::leith(S(0), S(1), S(2), S(3), J, P, Q);
              S(0) = J; S(1) = P; S(2) = Q;
            } else if constexpr (PROG == RP_SMAG) {
              T J, P, Q;
              PtProducts<T>::smag(S(0), S(1), S(2), S(3), S(4), S(5), J, P, Q);
              S(0) = J; S(1) = P; S(2) = Q;
            } else if constexpr (PROG == RP_DLEITH) {
              T J, P, Q, Jt, Pt, Qt;
              PtProducts<T>::leith(S(0), S(1), S(2), S(3), J, P, Q);
              PtProducts<T>::leith(S(4), S(5), S(6), S(7), Jt, Pt, Qt);
              S(0) = J; S(1) = P; S(2) = Q; S(3) = Jt; S(4) = Pt; S(5) = Qt;
            } else if constexpr (PROG == RP_DSMAG) {
              T J, P, Q, Jt, Pt, Qt;
              PtProducts<T>::smag(S(0), S(1), S(2), S(3), S(4), S(5), J, P, Q);
              PtProducts<T>::smag(S(6), S(7), S(8), S(9), S(10), S(11), Jt, Pt, Qt);
              S(0) = J; S(1) = P; S(2) = Q; S(3) = Jt; S(4) = Pt; S(5) = Qt;
            } else if constexpr (PROG == RP_ADJ_FWD) {
              // one stage recomputed for its adjoint: its fields kept as physical arrays, then the products
              const int kind = d.adj_kind;
              const T u = S(0), v = S(1), wx = S(2), wy = S(3);
              QG_ST(reinterpret_cast<T*>(d.pf[0]), px, n_phys, st, u);
              QG_ST(reinterpret_cast<T*>(d.pf[1]), px, n_phys, st, v);
              QG_ST(reinterpret_cast<T*>(d.pf[2]), px, n_phys, st, wx);
              QG_ST(reinterpret_cast<T*>(d.pf[3]), px, n_phys, st, wy);
              T J, P, Q;
              if (kind == 1) {
                const T pxy = S(4), pd = S(5);
                QG_ST(reinterpret_cast<T*>(d.pf[4]), px, n_phys, st, pxy);
                QG_ST(reinterpret_cast<T*>(d.pf[5]), px, n_phys, st, pd);
                PtProducts<T>::smag(u, v, wx, wy, pxy, pd, J, P, Q);
              } else {
                PtProducts<T>::leith(u, v, wx, wy, J, P, Q);
              }
              S(0) = J;
              if (kind != 0) {
                S(1) = P;
                S(2) = Q;
              }
            } else if constexpr (PROG == RP_ADJ_REV) {
              // transposed products of one stage (the linearisation of Eq. 1, 9, 10, 13): the adjoint field lam
              // and p = -lam_x, q = -lam_y against the kept fields
              const int kind = d.adj_kind;
              const T lam = S(0), p = -S(1), q = -S(2);
              const T wx = QG_LD(reinterpret_cast<const T*>(d.pf[2]), px, n_phys, st);
              const T wy = QG_LD(reinterpret_cast<const T*>(d.pf[3]), px, n_phys, st);
              S(0) = lam * wx;
              S(1) = lam * wy;
              S(2) = lam * QG_LD(reinterpret_cast<const T*>(d.pf[0]), px, n_phys, st);
              S(3) = lam * QG_LD(reinterpret_cast<const T*>(d.pf[1]), px, n_phys, st);
              if (kind != 0) {
                const T s2 = p * wx + q * wy;
                if (kind == 1) {
                  const T pxy = QG_LD(reinterpret_cast<const T*>(d.pf[4]), px, n_phys, st);
                  const T pd = QG_LD(reinterpret_cast<const T*>(d.pf[5]), px, n_phys, st);
                  const T gg = sqrt(T(4) * pxy * pxy + pd * pd);
                  const T ig = gg > T(0) ? T(1) / gg : T(0);
                  S(4) = gg * p;
                  S(5) = gg * q;
                  S(6) = T(4) * s2 * pxy * ig;
                  S(7) = s2 * pd * ig;
                } else {
                  const T gg = sqrt(wx * wx + wy * wy);
                  const T ig = gg > T(0) ? T(1) / gg : T(0);
                  S(4) = gg * p + s2 * wx * ig;
                  S(5) = gg * q + s2 * wy * ig;
                }
              }
            }
            if (d.check_finite) {
              constexpr int no = PROG == RP_NONE ? 1 : PROG == RP_DLEITH || PROG == RP_DSMAG ? 6 : 3;  // of a step's programs
#pragma unroll
              for (int i = 0; i < no; ++i) bad |= nonfinite(S(i));
            }
#undef S
          }
          __syncthreads();
        }
      } else if constexpr (PROG == RP_SCALE) {
        // Brinkman (two fields) or sponge (one field): multiply by the exact factor field
        const T* fac = reinterpret_cast<const T*>(d.factor);
        if (on) {
#pragma unroll
          for (int m = 0; m < EL; ++m) {
            const int k = t + sh.tt() * m;
            const T f0 = QG_LD(fac, ya * N + k, n_phys, st);
            const T f1 = two ? QG_LD(fac, yb * N + k, n_phys, st) : T(0);
            x[m] = mk<C>(x[m].y * f0, x[m].x * f1);
            bad |= nonfinite(x[m].x) | nonfinite(x[m].y);
          }
        }
      } else if (on) {  // RP_COPY to physical rows
        const bool batch = d.npair > 0;
        T* pa = reinterpret_cast<T*>(batch ? d.pout[k2.fa] : k2.fa ? d.phys_out2 : d.phys_out);
        T* pb = reinterpret_cast<T*>(batch ? d.pout[k2.fb] : k2.fb ? d.phys_out2 : d.phys_out);
#pragma unroll
        for (int m = 0; m < EL; ++m) {
          const int k = t + sh.tt() * m;
          QG_ST(pa, ya * N + k, n_phys, st, x[m].y);
          if (two) QG_ST(pb, yb * N + k, n_phys, st, x[m].x);
        }
      }
    } else {
      // split the transform of two real rows into their half spectra, optional i k_x, store the kept columns
      C* ub = fb.take();
      if (fb.active) {
#pragma unroll
        for (int m = 0; m < EL; ++m) QG_ST(ub, t + sh.tt() * m, fb.len, st, x[m]);
      }
      fb.sync();
      if (on) {
        C* A = reinterpret_cast<C*>(d.out[k2.fa]);
        C* B = reinterpret_cast<C*>(d.out[k2.fb]);
        const bool dxa = (d.dx_mask >> k2.fa) & 1u, dxb = (d.dx_mask >> k2.fb) & 1u;
#pragma unroll
        for (int m = 0; m < EL; ++m) {
          const int k = t + sh.tt() * m;
          if (k < g.Kcp) {
            C a = mk<C>(T(0), T(0)), b = mk<C>(T(0), T(0));
            if (k < g.Kc) {
              const C z = x[m];
              const C zm = QG_LD(ub, k == 0 ? 0 : N - k, fb.len, st);
              a = mk<C>(T(0.5) * (z.x + zm.x), T(0.5) * (z.y - zm.y));
              b = mk<C>(T(0.5) * (z.y + zm.y), T(-0.5) * (z.x - zm.x));
              const T kx = wavenumber<T>(g, k);
              if (dxa) a = cmul_ik(a, kx);
              if (dxb) b = cmul_ik(b, kx);
            }
            QG_ST(A, ya * g.IP + k, n_mixed, st, a);
            if (two) QG_ST(B, yb * g.IP + k, n_mixed, st, b);
          }
        }
      }
    }
  }
  if (d.check_finite && d.flag) {
    if (__syncthreads_or(bad) && tid == 0) atomicOr(d.flag, 1);
  }
}

template <typename T, class Sh>
cudaError_t launch_row_shape(const Geom& g, const FftPlan& plan, const Sh& sh, const RowDesc& d, const void* tw,
                             cudaStream_t st) {
  const RowConfig c = row_config(plan, d, (int)sizeof(T));
  const auto* twp = reinterpret_cast<const cplx_t<T>*>(tw);
  const dim3 grid(c.full + (g.n - c.full * c.rows)), block(c.threads);
#define QG_ROW_P(P)                                                           \
  case P: {                                                                   \
    const cudaError_t e = raise_smem_limit<row_kernel<T, Sh, P>>(c.smem);     \
    if (e != cudaSuccess) return e;                                           \
    return launch_pdl(d.pdl != 0, row_kernel<T, Sh, P>, grid, block, c.smem, st, g, sh, c, d, twp); \
  }
  switch (d.prog) {
    QG_ROW_P(RP_NONE)
    QG_ROW_P(RP_LEITH)
    QG_ROW_P(RP_SMAG)
    QG_ROW_P(RP_DLEITH)
    QG_ROW_P(RP_DSMAG)
    QG_ROW_P(RP_SCALE)
    QG_ROW_P(RP_COPY)
    QG_ROW_P(RP_ADJ_FWD)
    QG_ROW_P(RP_ADJ_REV)
  }
#undef QG_ROW_P
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_row(const Geom& g, const FftPlan& plan, const RowDesc& d, const void* tw, cudaStream_t st) {
  switch (plan.el) {
    case 4: return launch_row_shape<T>(g, plan, RtShape<4>{plan}, d, tw, st);
    case 8: return launch_row_shape<T>(g, plan, RtShape<8>{plan}, d, tw, st);
    case 12: return launch_row_shape<T>(g, plan, RtShape<12>{plan}, d, tw, st);
    case 18: return launch_row_shape<T>(g, plan, RtShape<18>{plan}, d, tw, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace qg
