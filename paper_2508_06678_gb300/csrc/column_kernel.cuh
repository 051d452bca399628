// Column pass: one CTA owns W adjacent k_x columns over the whole k_y / y
// range.  It forward y-transforms the mixed arrays produced by a row pass,
// does all spectral-space work of the step for its columns, and inverse
// y-transforms the fields the next row pass needs.
//
// Spectral-space work (Sec. II-A..E, III-A):
//   psi_hat = -w_hat / |k|^2, psi_hat(0) = 0                 (Eq. 1)
//   L = -J_hat - beta i k_x psi_hat + C D_hat                (Eq. 1, 9)
//   D_hat = i k_x F[g w_x] + i k_y F[g w_y]   (i k_x applied by the row pass)
//   SSP-RK3 stage  w_{s+1} = a w_0 + b (w_s + dt L)
//   Germano / Lilly (Eq. 12, 14): H = J~ - G J, M = r^p D~ - G D,
//     partial sums of sum_k w_k Re(H conj M) and w_k |M|^2 (w_k = 1 on k_x = 0,
//     else 2) in FP64 per CTA; C = max(0, <HM>/<MM>) (0 if <MM> = 0)
//   viscous/friction factor exp(-(nu|k|^2 + mu) dt) (exact)
//   Brinkman curl w = i k_x v_hat - i k_y u_hat (Eq. 2)
// Every output is confined to the 2/3 band by construction (only kept modes
// are stored).
#pragma once

#include "fft.cuh"
#include "qg_kernels.h"
#include "spectral.cuh"

namespace qg {

// A CTA's groups of TT threads transform c.fields fields of its W columns side by side (thread = (field, position,
// column), columns fastest so that a warp's accesses to a row of the mixed arrays are adjacent).  With one field at
// a time every thread keeps to its own modes and the partial results stay where it wrote them; with several, the
// transforms meet in shared memory, a thread then taking one mode of every field: a small grid has too few columns
// to fill the chip, and a pass is as long as one column's chain of transforms.  The state and its streamfunction
// (both over N^2) wait in shared memory for the derived fields, so 1 / |k|^2 is formed once per mode.
template <typename T, class Sh, int OP>
__global__ void __launch_bounds__(pass_threads(Sh::EL, sizeof(T))) col_kernel(Geom g, Sh sh, ColConfig cf, ColDesc d,
                                                                 const __grid_constant__ ColScalars<T> cs,
                                                                 const cplx_t<T>* __restrict__ twg) {
  using C = cplx_t<T>;
  constexpr int EL = Sh::EL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[2][32];
  __shared__ int dlist[kMaxDer];
  const int N = sh.n(), K = sh.band(g), Ny = 2 * K + 1, W = cf.w, F = cf.fields;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int nbuf = cf.one_buf ? 1 : 2;
  const int cp = cf.pitch;  // complex elements of one exchange buffer
  C* const tws = reinterpret_cast<C*>(smem_raw);
  C* const bufs = tws + (tw_shared(sh.table()) ? sh.table() : 0);
  const C* tw = tw_stage(twg, sh.table(), tws);
  pdl_enter();
  const int stop = d.flag ? *reinterpret_cast<volatile int*>(d.flag) : 0;
  C* const slotA = bufs + (size_t)F * W * nbuf * cp;  // [W][Ny]
  C* const slotB = slotA + (size_t)W * Ny;            // [W][Ny]
  // this CTA's column tile and its part of the tile's outgoing fields
  const int over = (int)blockIdx.x - cf.full;
  const int tile = over < 0 ? blockIdx.x : cf.full + over / cf.split;
  const int part = over < 0 ? 0 : over % cf.split, nparts = over < 0 ? 1 : cf.split;
  const int c0 = tile * W;
  const int nspec = W * Ny;
  // extents for the bounds-checked debug build
  int* const st = d.err;
  const long long n_mixed = (long long)N * g.IP, n_spec = (long long)g.Kcp * g.SP;
  const long long n_part = 2LL * gridDim.x;  // Germano partial sums: two per column CTA
  (void)n_mixed; (void)n_spec; (void)n_part; (void)st;

  // this thread's group: field slot fl, column c, position t
  const int fl = tid / (sh.tt() * W);
  const int in_f = tid - fl * sh.tt() * W;
  const int t = in_f / W, c = in_f - t * W;
  FftBufs<C> fb;
  fb.active = fl < F;
  fb.one = cf.one_buf;
  fb.warp = cf.warp;
  fb.st = st;
  fb.len = cp;
  const int slot = fb.active ? fl * W + c : 0;
  // the buffers of one parity lie together, so that adjacent columns keep their bank offset
  fb.b[0] = bufs + (size_t)slot * cp;
  fb.b[1] = cf.one_buf ? fb.b[0] : bufs + (size_t)(F * W + slot) * cp;

  C* w0 = reinterpret_cast<C*>(d.w0);
  C* ws = reinterpret_cast<C*>(d.ws);
  C* jh = reinterpret_cast<C*>(d.jh);
  C* dh = reinterpret_cast<C*>(d.dh);
  const T rpow = cs.rpow;
  const T inv_eta = cs.inv_eta;
  GermanoAcc<T> acc_hm, acc_mm;

  // mode r of column cc in the forward transform X of field f: what the op keeps of it
  auto accumulate = [&](int f, int cc, int r, C X) {
    const int e = cc * Ny + r;
    const int mx = c0 + cc;
    const int my = my_of_r(g, r);
    if (mx >= g.Kc) X = mk<C>(T(0), T(0));
    const T ky = wavenumber<T>(g, my), kx = wavenumber<T>(g, mx);
    const int gi = mx * g.SP + r;
    switch (OP) {
      case CO_STAGE_STATIC:
        if (f == 0) QG_ST(slotA, e, nspec, st, mk<C>(-X.x, -X.y));                                 // -J
        else if (f == 1) QG_ST(slotB, e, nspec, st, X);                                            // i kx F[g wx]
        else QG_ST(slotB, e, nspec, st, cadd(QG_LD(slotB, e, nspec, st), cmul_ik(X, ky)));         // + i ky F[g wy]
        break;
      case CO_DYN_REDUCE: {
        const bool in_test = mx * mx + my * my <= d.test_m2max;
        if (f == 0) {                                              // J
          QG_ST(slotA, e, nspec, st, X);
          QG_ST(jh, gi, n_spec, st, X);
        } else if (f == 1) {                                       // i kx F[g wx]
          QG_ST(slotB, e, nspec, st, X);
        } else if (f == 2) {                                       // D = .. + i ky F[g wy]
          const C D = cadd(QG_LD(slotB, e, nspec, st), cmul_ik(X, ky));
          QG_ST(dh, gi, n_spec, st, D);
          QG_ST(slotB, e, nspec, st, in_test ? mk<C>(-D.x, -D.y) : mk<C>(T(0), T(0)));             // -G D
        } else if (f == 3) {                                       // H = J~ - G J
          QG_ST(slotA, e, nspec, st, in_test ? csub(X, QG_LD(slotA, e, nspec, st)) : X);
        } else if (f == 4) {                                       // M = r^p D~ - G D
          QG_ST(slotB, e, nspec, st, cadd(QG_LD(slotB, e, nspec, st), cscale(X, rpow)));
        } else if (f == 6) {  // Brinkman pair of the paper's scheme: F_obs = (i ky F[chi u] - i kx F[chi v]) / eta
          QG_ST(slotA, e, nspec, st, cscale(cmul_ik(X, ky), inv_eta));
        } else if (f == 7) {
          const C Fo = csub(QG_LD(slotA, e, nspec, st), cscale(cmul_ik(X, kx), inv_eta));
          QG_ST(reinterpret_cast<C*>(d.bh), gi, n_spec, st, Fo);
        } else {
          const C M = cadd(QG_LD(slotB, e, nspec, st), cscale(cmul_ik(X, ky), rpow));
          const C H = QG_LD(slotA, e, nspec, st);
          const T wgt = mx == 0 ? T(1) : T(2);
          if (mx < g.Kc) {
            acc_hm.add_prod(wgt * H.x, M.x);
            acc_hm.add_prod(wgt * H.y, M.y);
            acc_mm.add_prod(wgt * M.x, M.x);
            acc_mm.add_prod(wgt * M.y, M.y);
          }
        }
        break;
      }
      case CO_CURL:
        if (f == 0) QG_ST(slotA, e, nspec, st, X);                                                       // u
        else QG_ST(slotA, e, nspec, st, csub(cmul_ik(X, kx), cmul_ik(QG_LD(slotA, e, nspec, st), ky)));  // i kx v - i ky u
        break;
      case CO_AB2CN:  // E = -J + C D + F_obs: slot A collects -J + F_obs, slot B collects D
        if (f == 0) QG_ST(slotA, e, nspec, st, mk<C>(-X.x, -X.y));
        else if (f < d.nst) QG_ST(slotB, e, nspec, st, (f == 1) ? X : cadd(QG_LD(slotB, e, nspec, st), cmul_ik(X, ky)));
        else if (f == d.nst) QG_ST(slotA, e, nspec, st, cadd(QG_LD(slotA, e, nspec, st), cscale(cmul_ik(X, ky), inv_eta)));
        else QG_ST(slotA, e, nspec, st, csub(QG_LD(slotA, e, nspec, st), cscale(cmul_ik(X, kx), inv_eta)));
        break;
      case CO_FORWARD2:
        if (f == 0) QG_ST(slotA, e, nspec, st, X);
        else QG_ST(slotB, e, nspec, st, X);
        break;
      case CO_FORWARD_N:  // field f's band straight to its own spectral array
        if (mx < g.Kc)
          QG_ST(reinterpret_cast<C*>(d.fout[f]), gi, n_spec, st,
                (d.zero_mean && mx == 0 && my == 0) ? mk<C>(T(0), T(0)) : X);
        break;
      default:  // CO_FORWARD, CO_AB2CN_FINAL
        QG_ST(slotA, e, nspec, st, X);
        break;
    }
  };

  C x[EL];
#pragma unroll
  for (int m = 0; m < EL; ++m) x[m] = mk<C>(T(0), T(0));
  // the derived fields this CTA's columns need: test-filtered fields vanish for k_x beyond the test band, and their
  // arrays stay zero there
  int nder = 0;
  for (int q = 0; q < d.nder; ++q) {
    if (((d.der[q] & D_TEST) && c0 > d.test_kmax) || q % nparts != part) continue;
    if (tid == 0) dlist[nder] = q;
    ++nder;
  }
  const int nfr = (d.nfwd + F - 1) / F, nir = (nder + F - 1) / F;
#pragma unroll 1
  for (int it = 0; it <= nfr + nir; ++it) {
    if (it == nfr) {
      if constexpr (OP == CO_FORWARD_N) return;  // every field's band is stored
      T coeff = cs.coeff;
      if constexpr (OP == CO_DYN_COMBINE || OP == CO_AB2CN_COMBINE) {
        if (!germano_coefficient(d.partials, d.npartials, red, nt, stop, d.coeff_out, st)) return;
        coeff = T(red[0][0]);
      } else if (__syncthreads_or(nfr == 0 ? stop : 0)) {  // also completes the slots and dlist
        return;
      }
      if constexpr (OP == CO_DYN_REDUCE) {
        // the CTA's Germano partial sums
        pair_sum(acc_hm.value(), acc_mm.value(), red, (nt + 31) >> 5);
        if (tid == 0) {
          QG_ST(d.partials, 2LL * blockIdx.x, n_part, st, red[0][0]);
          QG_ST(d.partials, 2LL * blockIdx.x + 1, n_part, st, red[1][0]);
        }
        return;
      }

      // ---- new vorticity spectrum for the owned columns.  The modes go in batches whose global loads are all
      // issued before any of the batch's stores: the state arrays may alias as far as the compiler can tell, so a
      // load placed after a store would wait for that store's round trip.
      const T dt = cs.dt, a_rk = cs.a, b_rk = cs.b, beta = cs.beta;
      const T* vx = reinterpret_cast<const T*>(d.visc_x);
      const T* vy = reinterpret_cast<const T*>(d.visc_y);
      const T vmu = cs.visc_mu, scale = cs.scale;
      const T* ik2t = reinterpret_cast<const T*>(d.ik2);
      const C* bhp = reinterpret_cast<const C*>(d.bh);
      C* ep = reinterpret_cast<C*>(d.eprev);
      C* wsp = reinterpret_cast<C*>(d.wss);
      constexpr int GB = 4;
      for (int e0 = tid; e0 < nspec; e0 += GB * nt) {
        // per op: u0 = w^n (or w* in the AB2CN final), u1 = stage field or E_prev, u2 = J, u3 = D, u4 = Brinkman
        // forcing, u5 = previous w*; vf = viscous factor
        C u0[GB], u1[GB], u2[GB], u3[GB], u4[GB], u5[GB];
        T vf[GB], ik[GB];
#pragma unroll
        for (int q = 0; q < GB; ++q) {
          const int e = e0 + q * nt;
          const C z = mk<C>(T(0), T(0));
          u0[q] = z; u1[q] = z; u2[q] = z; u3[q] = z; u4[q] = z; u5[q] = z;
          vf[q] = T(1);
          ik[q] = T(0);
          const int cc = e / Ny, r = e - cc * Ny, mx = c0 + cc;
          if (e < nspec && mx < g.Kc) {
            const int gi = mx * g.SP + r;
            switch (OP) {
              case CO_DERIVE: u0[q] = QG_LD(w0, gi, n_spec, st); break;
              case CO_STAGE_STATIC:
              case CO_DYN_COMBINE:
                u0[q] = QG_LD(w0, gi, n_spec, st);
                u1[q] = d.use_ws ? QG_LD(ws, gi, n_spec, st) : u0[q];
                if (OP == CO_DYN_COMBINE) {
                  u2[q] = QG_LD(jh, gi, n_spec, st);
                  u3[q] = QG_LD(dh, gi, n_spec, st);
                }
                break;
              case CO_AB2CN:
              case CO_AB2CN_COMBINE:
                u0[q] = QG_LD(w0, gi, n_spec, st);
                if (OP == CO_AB2CN_COMBINE) {
                  u2[q] = QG_LD(jh, gi, n_spec, st);
                  u3[q] = QG_LD(dh, gi, n_spec, st);
                  if (d.brink) u4[q] = QG_LD(bhp, gi, n_spec, st);
                }
                if (!d.ab2_first) {
                  u1[q] = QG_LD(ep, gi, n_spec, st);
                  if (d.sponge_next) u5[q] = QG_LD(wsp, gi, n_spec, st);
                }
                break;
              case CO_AB2CN_FINAL: u0[q] = QG_LD(wsp, gi, n_spec, st); break;
              default: break;
            }
            // FP64: 1 / |k|^2 from the handle's table (a division is some ten FP64 operations a mode)
            const int my = my_of_r(g, r);
            ik[q] = sizeof(T) == 8 && ik2t ? QG_LD(ik2t, gi, n_spec, st) : inv_k2<T>(cs, mx * mx + my * my);
            if (d.viscous) vf[q] = QG_LD(vx, mx, g.Kcp, st) * QG_LD(vy, r, g.SP, st) * vmu;
          }
        }
#pragma unroll
        for (int q = 0; q < GB; ++q) {
          const int e = e0 + q * nt;
          if (e >= nspec) continue;
          const int cc = e / Ny, r = e - cc * Ny, mx = c0 + cc;
          const int my = my_of_r(g, r);
          const int m2 = mx * mx + my * my;
          const int gi = mx * g.SP + r;
          C wn = mk<C>(T(0), T(0));
          const T ik2 = ik[q];
          if (mx < g.Kc) {
            switch (OP) {
              case CO_DERIVE:
                wn = u0[q];
                break;
              case CO_STAGE_STATIC:
              case CO_DYN_COMBINE: {
                const C wz = u0[q], wst = u1[q];
                const C psi = mk<C>(-wst.x * ik2, -wst.y * ik2);
                const T kx = wavenumber<T>(g, mx);
                const C bv = cscale(cmul_ik(psi, kx), beta);
                C Lw;
                if (OP == CO_STAGE_STATIC) {
                  Lw = csub(QG_LD(slotA, e, nspec, st), bv);
                  if (d.nfwd > 1) Lw = cadd(Lw, cscale(QG_LD(slotB, e, nspec, st), coeff));
                } else {
                  Lw = csub(mk<C>(-u2[q].x, -u2[q].y), bv);
                  Lw = cadd(Lw, cscale(u3[q], coeff));
                }
                const C inner = cadd(wst, cscale(Lw, dt));
                wn = cadd(cscale(wz, a_rk), cscale(inner, b_rk));
                break;
              }
              case CO_AB2CN:
              case CO_AB2CN_COMBINE: {
                // Eq. 4: w* = ((1 + dt/2 lin) w^t + dt (3/2 E - 1/2 E_prev)) / (1 - dt/2 lin)
                C E;
                if (OP == CO_AB2CN) {
                  E = QG_LD(slotA, e, nspec, st);
                  if (d.nst > 1) E = cadd(E, cscale(QG_LD(slotB, e, nspec, st), coeff));
                } else {
                  E = cadd(mk<C>(-u2[q].x, -u2[q].y), cscale(u3[q], coeff));
                  if (d.brink) E = cadd(E, u4[q]);
                }
                const C Ep = d.ab2_first ? E : u1[q];
                QG_ST(ep, gi, n_spec, st, E);
                const T k2 = cs.ks2 * T(m2);
                const T kx = wavenumber<T>(g, mx);
                const T hdt = T(0.5) * dt;
                const T lre = -(cs.nu * k2 + cs.mu);
                const T lim = beta * kx * ik2;
                const C wz = u0[q];
                const C ab = mk<C>(T(1.5) * E.x - T(0.5) * Ep.x, T(1.5) * E.y - T(0.5) * Ep.y);
                const C num = cadd(cmul(mk<C>(T(1) + hdt * lre, hdt * lim), wz), cscale(ab, dt));
                const T dre = T(1) - hdt * lre, dim = -hdt * lim;
                const T den = dre * dre + dim * dim;
                const C wst = mk<C>((num.x * dre + num.y * dim) / den, (num.y * dre - num.x * dim) / den);
                if (d.sponge_next) {
                  const C wss = d.ab2_first ? wst : u5[q];
                  QG_ST(wsp, gi, n_spec, st, wst);
                  wn = mk<C>(T(1.5) * wst.x - T(0.5) * wss.x, T(1.5) * wst.y - T(0.5) * wss.y);
                } else {
                  wn = wst;
                }
                break;
              }
              case CO_AB2CN_FINAL:
                wn = csub(u0[q], QG_LD(slotA, e, nspec, st));
                break;
              default:  // CO_CURL, CO_FORWARD, CO_FORWARD2
                wn = QG_LD(slotA, e, nspec, st);
                break;
            }
            if (d.viscous) wn = cscale(wn, vf[q]);
            if (d.zero_mean && m2 == 0) wn = mk<C>(T(0), T(0));
            if (d.store_ws && part == 0) QG_ST(reinterpret_cast<C*>(d.ws_out), gi, n_spec, st, wn);
            if (d.store_w0 && part == 0) QG_ST(w0, gi, n_spec, st, wn);
            if (OP == CO_FORWARD2) {  // the second field, treated like the first
              C wb = QG_LD(slotB, e, nspec, st);
              if (d.viscous) wb = cscale(wb, vf[q]);
              if (d.zero_mean && m2 == 0) wb = mk<C>(T(0), T(0));
              QG_ST(reinterpret_cast<C*>(d.w0b), gi, n_spec, st, wb);
            }
          }
          if (nder > 0) {
            if constexpr (sizeof(T) == 8 && EL % 3 == 0)  // N has factors of 3
              wn = mk<C>(fma(wn.x, scale, wn.x * cs.scale_lo), fma(wn.y, scale, wn.y * cs.scale_lo));
            else
              wn = cscale(wn, scale);
            QG_ST(slotA, e, nspec, st, wn);
            QG_ST(slotB, e, nspec, st, mk<C>(-wn.x * ik2, -wn.y * ik2));
          }
        }
      }
      if (nir == 0) return;
      __syncthreads();
    }
    if (it == nfr + nir) return;
    const bool fwd = it < nfr;
    const int f = fwd ? it * F + fl : (it - nfr) * F + fl;
    const bool on = fb.active && f < (fwd ? d.nfwd : nder);
    const int mx = c0 + c;
    int q = 0;

    // ---- the transform's input: a mixed array's columns, or a derived field of the new state
    if (on && fwd) {
      const C* src = reinterpret_cast<const C*>(d.fin[f]);
#pragma unroll
      for (int m = 0; m < EL; ++m)
        x[m] = QG_LD(src, (t + sh.tt() * m) * g.IP + mx, n_mixed, st);
    } else if (on) {
      q = dlist[f];
      const int code = d.der[q];
      const T kx = wavenumber<T>(g, mx);
      const bool psi = (code & 7) == D_U || (code & 7) == D_V || (code & 7) == D_PXY || (code & 7) == D_PD;
      const C* sl = psi ? slotB : slotA;
#pragma unroll
      for (int m = 0; m < EL; ++m) {
        const int k = t + sh.tt() * m;
        C v = mk<C>(T(0), T(0));
        if (k <= K || k >= N - K) {
          const int my = k <= K ? k : k - N;
          const T ky = wavenumber<T>(g, my);
          if (!(code & D_TEST) || mx * mx + my * my <= d.test_m2max) {
            const C s = QG_LD(sl, c * Ny + (k <= K ? k : k - N + Ny), nspec, st);
            switch (code & 7) {
              case D_U: v = cmul_ik(s, -ky); break;                       // -d psi / dy (+ U)
              case D_V: v = cmul_ik(s, kx); break;                        // d psi / dx
              case D_WX: v = cmul_ik(s, kx); break;
              case D_WY: v = cmul_ik(s, ky); break;
              case D_PXY: v = cscale(s, -(kx * ky)); break;
              case D_PD: v = cscale(s, -(kx * kx - ky * ky)); break;
              default: v = s; break;
            }
          }
          if ((code & 7) == D_U && mx == 0 && my == 0) v = mk<C>(cs.U, T(0));
        }
        x[m] = mk<C>(v.y, v.x);
      }
    }

    // the status flag's load has overlapped the inputs'; the barrier also completes the twiddle table
    if (it == 0 && fwd && __syncthreads_or(stop)) return;
    sh.run(x, t, fb, tw);

    if (!fwd) {
      if (on) {
        C* dst = reinterpret_cast<C*>(d.dout[q]);
#pragma unroll
        for (int m = 0; m < EL; ++m)
          QG_ST(dst, (t + sh.tt() * m) * g.IP + mx, n_mixed, st, mk<C>(x[m].y, x[m].x));
      }
    } else if (F == 1) {
      if (on) {
#pragma unroll
        for (int m = 0; m < EL; ++m) {
          const int k = t + sh.tt() * m;
          if (k <= K || k >= N - K) accumulate(f, c, k <= K ? k : k - N + Ny, x[m]);
        }
      }
    } else {
      C* out = fb.take();
      if (fb.active) {
#pragma unroll
        for (int m = 0; m < EL; ++m) QG_ST(out, t + sh.tt() * m, fb.len, st, x[m]);
      }
      __syncthreads();
      const int par = cf.one_buf ? 0 : fb.ph ^ 1;  // parity of the tiles' buffers
      const C* tiles = bufs + (size_t)par * F * W * cp;
      const int f1 = min(d.nfwd - it * F, F);
      for (int e = tid; e < nspec; e += nt) {
        const int cc = e / Ny, r = e - cc * Ny;
        for (int s = 0; s < f1; ++s)
          accumulate(it * F + s, cc, r, QG_LD(tiles, (s * W + cc) * cp + row_of_r(g, r), F * W * cp, st));
      }
      __syncthreads();
    }
  }
}

template <typename T, class Sh>
cudaError_t launch_col_shape(const Geom& g, const FftPlan& plan, const Sh& sh, const ColDesc& d, const void* tw, int W,
                             cudaStream_t st) {
  const ColConfig c = col_config(g, plan, d, W, (int)sizeof(T));
  const auto* twp = reinterpret_cast<const cplx_t<T>*>(tw);
  const dim3 grid(c.grid), block(c.threads);
  const ColScalars<T> cs = col_scalars<T>(g, d);
#define QG_COL_P(P)                                                           \
  case P: {                                                                   \
    const cudaError_t e = raise_smem_limit<col_kernel<T, Sh, P>>(c.smem);     \
    if (e != cudaSuccess) return e;                                           \
    return launch_pdl(d.pdl != 0, col_kernel<T, Sh, P>, grid, block, c.smem, st, g, sh, c, d, cs, twp); \
  }
  switch (d.op) {
    QG_COL_P(CO_DERIVE)
    QG_COL_P(CO_STAGE_STATIC)
    QG_COL_P(CO_DYN_REDUCE)
    QG_COL_P(CO_DYN_COMBINE)
    QG_COL_P(CO_CURL)
    QG_COL_P(CO_FORWARD)
    QG_COL_P(CO_AB2CN)
    QG_COL_P(CO_AB2CN_COMBINE)
    QG_COL_P(CO_AB2CN_FINAL)
    QG_COL_P(CO_FORWARD2)
    QG_COL_P(CO_FORWARD_N)
  }
#undef QG_COL_P
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_col(const Geom& g, const FftPlan& plan, const ColDesc& d, const void* tw, int W, cudaStream_t st) {
  switch (plan.el) {
    case 4: return launch_col_shape<T>(g, plan, RtShape<4>{plan}, d, tw, W, st);
    case 8: return launch_col_shape<T>(g, plan, RtShape<8>{plan}, d, tw, W, st);
    case 12: return launch_col_shape<T>(g, plan, RtShape<12>{plan}, d, tw, W, st);
    case 18: return launch_col_shape<T>(g, plan, RtShape<18>{plan}, d, tw, W, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace qg
