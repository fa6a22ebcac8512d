// Resident single-mode solver kernel: whole RK4 steps of Eqs. 9a-c with the system on chip.
//
// A group of warps loads one system's state, advances it n_steps steps in registers and shared
// memory and writes it back, so HBM sees four transfers per call (y and its compensation, in and
// out) instead of 18 per step.  A launch serves bq_step and bq_solve alike.
//
// Arithmetic per point (k, l) of R, with a(t) the coefficient of the left-hand term with source
// k - 1 (i h e(t) for a drive h e(t) a^dag + h.c.; the host checks that the three other
// off-diagonal terms are -conj(a), -a and conj(a), as they are for a Hermitian H):
//   d(k,l) u + a (xm_k u(k-1,l) - yp_l u(k,l+1)) - conj(a) (xp_k u(k+1,l) - ym_l u(k,l-1))
//   + sm_kl u(k-1,l-1) + sm_k G_x[k-1] sm_l G_y[l-1] + the same with +1
// The weights are real and static: they stay in registers for the whole call, and only a(t)
// changes with the stage (no per-stage coefficient vectors).  A purely imaginary a (a real
// envelope) needs 2 instead of 8 multiply-adds for the two products.
//
// What it replaces and measured (one GB300): the streamed step kernel was bound by HBM traffic
// and issue, the earlier persistent solve by issue (160 instructions per point and stage, most of
// them loads and rebuilding of per-stage coefficients).  4096 ragged FP32 oscillators (N 10..40):
// 84 -> 18.6 us per step; 16 384: 351 -> 79; 1024 in FP64: 413 -> 120; one in FP32 (N = 40):
// 14.2 -> 2.0; one in FP64: 145 -> 36.  What bounds it now: in FP32 shared-memory wavefronts and
// issue about equally (a half each, 20 warps per SM to hide the latencies); in FP64 the FP64 pipe
// (88%).
//
// Layout: a thread owns column l and RB consecutive rows, its state, stage sum, compensation,
// stage input and weights in registers; the column's own neighbours never leave registers, and
// the left and right columns are read once each from shared memory (the sandwich sources are
// the same values one row earlier).  Two stage buffers alternate; one barrier of the group per
// stage.  The group's last warp advances G_x, G_y and evaluates the envelope for eight steps
// (32 stages, one per lane) at a time.
//
// HERM: a Hermitian measured operator's system (p = q) stays Hermitian: R = R^dagger and
// G_y = conj(G_x).  With P the grid size rounded up to an odd number (the added index holds
// zeros), row d of the layout holds the elements (k, l), k = (l + d) mod P, for d = 0 .. D = P/2:
// every pair (k, l), (l, k) exactly once.  In this layout (k-1, l) is row d-1, (k, l+1) row d-1
// of column l+1, (k, l-1) row d+1 of column l-1 and (k-+1, l-+1) row d of the next column, so
// the same loop serves both layouts with the side columns' rows shifted by one; the rows beyond
// the ends are conjugates of stored ones (row -1, column l: conj of row 1, column l-1; row D+1:
// conj of row D, column (l+D+1) mod P).  Half the points, the same results to rounding.
#pragma once

#include "bq_device.cuh"
#include "bq_resident.h"

namespace bq {

__device__ __forceinline__ void group_sync(int id, int n) {
  asm volatile("barrier.cta.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Conjugate where m is the sign bit, unchanged where m is zero (integer pipe: FP64 is scarce).
__device__ __forceinline__ float2 conj_if(float2 v, unsigned m) {
  v.y = __uint_as_float(__float_as_uint(v.y) ^ m);
  return v;
}
__device__ __forceinline__ double2 conj_if(double2 v, unsigned m) {
  v.y = __hiloint2double(__double2hiint(v.y) ^ (int)m, __double2loint(v.y));
  return v;
}

// y + d exactly as (y, -comp), whichever of the two is larger.
template <typename C>
__device__ __forceinline__ void res_update(C d, C& y, C& c) {
  C t, e;
  sum_ordered(y, d, t, e);
  y = t;
  c = cneg(e);
}

// Products of the off-diagonal coefficient: a p - conj(a) q added to k.
template <int MODE, typename C>
__device__ __forceinline__ C off_diag(C a, C p, C q, C k) {
  if constexpr (MODE == 1) {  // a = i b
    const C s = cadd(p, q);
    k.x = fma(-a.y, s.y, k.x);
    k.y = fma(a.y, s.x, k.y);
  } else {
    C s, d;
    s.x = p.x + q.x; s.y = p.y + q.y;
    d.x = p.x - q.x; d.y = p.y - q.y;
    k.x = fma(a.x, d.x, fma(-a.y, s.y, k.x));
    k.y = fma(a.x, d.y, fma(a.y, s.x, k.y));
  }
  return k;
}

template <typename T>
__device__ __forceinline__ T res_const(const ResArgs& A, int i) {
  if constexpr (sizeof(T) == 8) return A.cd[i];
  else return A.cf[i];
}

template <typename T>
struct ResWeights {  // pointers into a problem's parameter block
  using C = typename C2T<T>::type;
  const C *dx, *dy;
  const T *xm, *xp, *ym, *yp, *smx, *smy, *spx, *spy;
  __device__ __forceinline__ ResWeights(const unsigned char* blk, int M) {
    dx = reinterpret_cast<const C*>(blk + sizeof(ResHdr));
    dy = dx + M;
    xm = reinterpret_cast<const T*>(dy + M);
    xp = xm + M; ym = xp + M; yp = ym + M;
    smx = yp + M; smy = smx + M; spx = smy + M; spy = spx + M;
  }
};

// What both roles of a group share: its pointers into shared and global memory.
template <typename T, int NS, bool HERM>
struct ResView {
  using C = typename C2T<T>::type;
  static constexpr int GW = HERM ? 1 : 2;  // G_x (and G_y) stored
  const unsigned char* blk;
  C *U, *Gs, *RG, *E, *yg, *cg;
  int M, P, ss, us, gt, gn, bar;
  bool sep;
  // U: [2] stage buffers of us elements, then the strips' compensation; the whole region is also the staging buffer of the load and the store.  Gs: [2][GW P] stage inputs of
  // G.  RG: [2][2][2 P] row products sm_k G_x[k-1], sp_k G_x[k+1] (HERM: twice, so that the
  // index l + d needs no modulo).  E: [2][32] off-diagonal coefficient of the stages.
  __device__ __forceinline__ ResView(const ResArgs& A, const ResGroup& g, unsigned char* sm, int gt_, int gn_, int bar_)
      : M(g.M), P(HERM ? g.M | 1 : g.M), gt(gt_), gn(gn_), bar(bar_) {
    blk = A.params + g.param_off;
    U = reinterpret_cast<C*>(sm);
    Gs = U + g.stage_elems;
    RG = Gs + 4 * P;
    E = RG + 8 * P;
    yg = reinterpret_cast<C*>(A.y) + g.blk_off;
    cg = reinterpret_cast<C*>(A.comp) + g.blk_off;
    ss = res_strip_stride(g.rb, P);
    us = g.nb * ss;
    sep = g.gy_off >= 0;
  }
  __device__ __forceinline__ void sync() const { group_sync(bar, gn); }
  __device__ __forceinline__ void stage_in(const C* src, int n) const {
    for (int i = gt; i < n; i += gn) U[i] = src[i];
    sync();
  }
  __device__ __forceinline__ void stage_out(C* dst, int n) const {
    sync();
    for (int i = gt; i < n; i += gn) dst[i] = U[i];
    sync();
  }
};

// The sequence of barriers of a group, the same for both roles: [y staged] [y taken] ([comp
// staged] [comp taken]) [ready], four per step, then [stage buffers free] [y placed] [y out]
// [comp placed] [comp out].

// The strips of R.
template <typename T, int RB, int MODE, int NS, bool SD, bool HERM>
__device__ __forceinline__ void res_strips(const ResArgs& A, const ResGroup& g, unsigned char* sm, int gt, int gn, int bar) {
  using C = typename C2T<T>::type;
  // registers are short: the compensation, touched once a step, lives in shared memory, and the
  // own stage input too except in the FP32 Hermitian layout
  constexpr bool US = sizeof(T) == 8 || !HERM;
  const ResView<T, NS, HERM> V(A, g, sm, gt, gn, bar);
  const ResWeights<T> W(V.blk, g.M);
  const int M = g.M, P = V.P, D = P / 2, ND = HERM ? D + 1 : M, us = V.us;
  C* U = V.U;
  const C zero = cmk<C>(0.0, 0.0);
  C* Cs = U + 2 * us + gt;  // this thread's compensation, row j at Cs[j nb P]
  const bool act = gt < g.nb * P;
  const int l = act ? gt % P : 0;
  // (the last strip may overlap the one before: both threads then compute the shared rows, with
  // explicit multiply-adds throughout so that they get the same bits, and store the same values)
  const int d0 = act ? min((gt / P) * RB, ND - RB) : 0;
  const bool first = HERM && d0 == 0, last = HERM && d0 + RB == ND;
  const unsigned m0 = first ? 0x80000000u : 0u, m1 = last ? 0x80000000u : 0u;
  const int lm = max(l - 1, 0), lp = min(l + 1, P - 1);  // (clamped columns have zero weights)
  // Element offsets in a stage buffer of the values around the strip.  Strip-major: strip b's rows
  // start at b SS, a row is S elements (a constant: the step from row to row is an immediate), and
  // SS is P modulo 16, so that the lanes of a half warp touch consecutive 8-byte banks across
  // strips too (a sixth fewer shared-memory wavefronts than plain rows).
  constexpr int S = BQ_RES_COLS;
  const int SS = V.ss;
  auto at = [&](int d) {  // row d, column 0 (rows the last two strips share: the last strip's copy)
    const int sb = d >= ND - RB ? g.nb - 1 : d / RB;
    return sb * SS + (d - min(sb * RB, ND - RB)) * S;
  };
  const int o_own = (act ? gt / P : 0) * SS + l;
  const int o_top = first ? at(1) + (l == 0 ? P - 1 : l - 1) : at(max(d0 - 1, 0)) + l;
  const int o_bot = last ? at(D) + (l + D + 1) % P : at(min(d0 + RB, ND - 1)) + l;
  const int o_lw = o_own - l + (HERM ? S : 0) + lm;  // left column at row j < RB - 1: o_lw + j S
  const int o_lend = last ? at(D) + (l + D) % P : (HERM ? at(d0 + RB) + lm : o_lw + (RB - 1) * S);
  const int o_lpre = HERM ? o_lw - S : at(max(d0 - 1, 0)) + lm;
  const int o_rw = o_own - l - (HERM ? S : 0) + lp;  // right column at row j > 0: o_rw + j S
  const int o_r0 = HERM ? (first ? at(1) + l : at(d0 - 1) + lp) : o_rw;
  const int o_rpost = HERM ? o_rw + RB * S : at(min(d0 + RB, M - 1)) + lp;
  const int k0 = HERM ? l + d0 : d0;  // row index of the first point (HERM: modulo P)
  auto row = [&](int j) { const int k = k0 + j; return HERM && k >= P ? k - P : k; };
  auto in = [&](int j) { return act && (!HERM || (l < M && row(j) < M)); };  // a point of the grid

  C y[RB], u[US ? 1 : RB], s[RB], dg[RB];
  T xm[RB], xp[RB], sm_[RB], sp_[NS == 2 ? RB : 1];
  V.stage_in(V.yg, g.blk_elems);
#pragma unroll
  for (int j = 0; j < RB; ++j) y[j] = in(j) ? U[g.r_off + row(j) * M + l] : zero;
  V.sync();
  {
    C ct[RB];
#pragma unroll
    for (int j = 0; j < RB; ++j) ct[j] = zero;
    if (!A.comp_zero) {
      V.stage_in(V.cg, g.blk_elems);
#pragma unroll
      for (int j = 0; j < RB; ++j)
        if (in(j)) ct[j] = U[g.r_off + row(j) * M + l];
      V.sync();
    }
#pragma unroll
    for (int j = 0; j < RB; ++j)
      if (act) Cs[j * g.nb * P] = ct[j];
  }
  const bool inl = l < M;
  const T ym = inl ? W.ym[l] : (T)0, yp = inl ? W.yp[l] : (T)0, smy = inl ? W.smy[l] : (T)0, spy = inl ? W.spy[l] : (T)0;
#pragma unroll
  for (int j = 0; j < RB; ++j) {
    const int k = row(j);
    const bool ok = in(j);
    dg[j] = ok ? cadd(W.dx[k], W.dy[l]) : zero;
    xm[j] = ok ? W.xm[k] : (T)0;
    xp[j] = ok ? W.xp[k] : (T)0;
    sm_[j] = ok ? W.smx[k] * smy : (T)0;
    if (NS == 2) sp_[j] = ok ? W.spx[k] * spy : (T)0;
    if (!US) u[US ? 0 : j] = y[j];
    if (act) U[o_own + j * S] = y[j];
    s[j] = zero;
  }
  V.sync();

  const T hh = res_const<T>(A, 0), h2 = res_const<T>(A, 1), w_hi = res_const<T>(A, 2), w_lo = res_const<T>(A, 3);

  // right-hand side at the strip's points from stage buffer B (half b of G), handed to f(j, k)
  auto rhs = [&](const C* B, int b, C a, auto f) {
    const C* G = V.Gs + b * V.GW * P;
    const C* r = V.RG + b * 4 * P + k0;
    C gl = G[(HERM ? 0 : P) + lm], gr = G[(HERM ? 0 : P) + lp];
    if (HERM) {
      gl = conj_if(gl, 0x80000000u);
      gr = conj_if(gr, 0x80000000u);
    }
    gl = cscale(gl, smy);
    gr = cscale(gr, spy);
    C up = conj_if(B[o_top], m0), lpre = B[o_lpre];
    C rj = conj_if(B[o_r0], m0);
    C uc = US ? B[o_own] : u[0];
#pragma unroll
    for (int j = 0; j < RB; ++j) {
      const C dn = j + 1 < RB ? (US ? B[o_own + (j + 1) * S] : u[US ? 0 : j + 1]) : conj_if(B[o_bot], m1);
      const C lj = j + 1 < RB ? B[o_lw + j * S] : conj_if(B[o_lend], m1);
      const C rn = j + 1 < RB ? B[o_rw + (j + 1) * S] : (NS == 2 ? B[o_rpost] : zero);
      C k, p, q;
      k.x = fma(dg[j].x, uc.x, -(dg[j].y * uc.y));
      k.y = fma(dg[j].x, uc.y, dg[j].y * uc.x);
      p.x = fma(xm[j], up.x, -yp * rj.x);
      p.y = fma(xm[j], up.y, -yp * rj.y);
      if constexpr (MODE == 1) {  // a = i b: p + q in one chain
        p.x = fma(xp[j], dn.x, fma(-ym, lj.x, p.x));
        p.y = fma(xp[j], dn.y, fma(-ym, lj.y, p.y));
        k.x = fma(-a.y, p.y, k.x);
        k.y = fma(a.y, p.x, k.y);
      } else {
        q.x = fma(xp[j], dn.x, -ym * lj.x);
        q.y = fma(xp[j], dn.y, -ym * lj.y);
        k = off_diag<MODE>(a, p, q, k);
      }
      // (SD, the secular projector: k = l only, in the Hermitian layout the first row)
      if (!SD || (HERM ? j == 0 && d0 == 0 : d0 + j == l)) {
        k = caxpy(sm_[j], lpre, k);
        k = cfma(r[j], gl, k);
        if constexpr (NS == 2) {
          k = caxpy(sp_[j], rn, k);
          k = cfma(r[2 * P + j], gr, k);
        }
      }
      if (HERM && j == 0 && d0 == 0) k.y = (T)0;  // the diagonal is real
      lpre = lj;
      rj = rn;
      up = uc;
      uc = dn;
      f(j, k);
    }
  };

  const int n_steps = A.n_steps;
#pragma unroll 1
  for (int step = 0; step < n_steps; ++step) {
    const C* Es = V.E + ((step >> 3) & 1) * 32 + (step & 7) * 4;
    // the state update of row j by the stage sum and k4
    auto update = [&](int j, C k) {
      C d, cj = Cs[j * g.nb * P];
      d.x = s[j].x + k.x;
      d.y = s[j].y + k.y;
      if constexpr (sizeof(T) == 4) {
        d.x = fma(w_hi, d.x, fma(w_lo, d.x, -cj.x));
        d.y = fma(w_hi, d.y, fma(w_lo, d.y, -cj.y));
      } else {  // (w_lo is zero)
        d.x = fma(w_hi, d.x, -cj.x);
        d.y = fma(w_hi, d.y, -cj.y);
      }
      res_update(d, y[j], cj);
      Cs[j * g.nb * P] = cj;
      s[j] = zero;
    };
    if constexpr (!US) {
      // One copy of the right-hand side for all four stages (the ragged batch runs several strip
      // lengths at once and would not fit the instruction caches with more): k replaces u row by
      // row, the combination follows.
#pragma unroll 1
      for (int stage = 1; stage <= 4; ++stage) {
        const int b = (stage & 1) ^ 1;  // stages 1, 3 read half 0; 2, 4 half 1
        if (act) {
          C* O = U + (b ^ 1) * us + o_own;
          rhs(U + b * us, b, Es[stage - 1], [&](int j, C k) { u[US ? 0 : j] = k; });
          if (stage < 4) {
            const T al = stage == 3 ? hh : h2, be = stage == 1 ? (T)1 : (T)2;
#pragma unroll
            for (int j = 0; j < RB; ++j) {
              C& v = u[US ? 0 : j];
              s[j] = caxpy(be, v, s[j]);
              v = caxpy(al, v, y[j]);
              O[j * S] = v;
            }
          } else {
#pragma unroll
            for (int j = 0; j < RB; ++j) {
              update(j, u[US ? 0 : j]);
              u[US ? 0 : j] = y[j];
              O[j * S] = y[j];
            }
          }
        }
        V.sync();
      }
    } else {
#pragma unroll 1
      for (int stage = 1; stage <= 3; ++stage) {
        const int b = (stage & 1) ^ 1;
        const T al = stage == 3 ? hh : h2, be = stage == 1 ? (T)1 : (T)2;
        if (act) {
          C* O = U + (b ^ 1) * us + o_own;
          rhs(U + b * us, b, Es[stage - 1], [&](int j, C k) {
            s[j] = caxpy(be, k, s[j]);
            O[j * S] = caxpy(al, k, y[j]);
          });
        }
        V.sync();
      }
      if (act) {
        C* O = U + o_own;
        rhs(U + us, 1, Es[3], [&](int j, C k) {
          update(j, k);
          O[j * S] = y[j];
        });
      }
      V.sync();
    }
  }

  // ---- store: through the staging buffer, coalesced ------------------------------------------
#pragma unroll
  for (int j = 0; j < RB; ++j) s[j] = act ? Cs[j * g.nb * P] : zero;
  V.sync();
  auto place = [&](int j, C v) {
    const int k = row(j);
    if (!in(j)) return;
    if (HERM) U[g.r_off + l * M + k] = conj_if(v, 0x80000000u);
    U[g.r_off + k * M + l] = v;
  };
#pragma unroll
  for (int j = 0; j < RB; ++j) place(j, y[j]);
  V.stage_out(V.yg, g.blk_elems);
#pragma unroll
  for (int j = 0; j < RB; ++j) place(j, s[j]);
  V.stage_out(V.cg, g.blk_elems);
}

// The group's last warp: G_x, G_y, the row products of the sandwich terms, the envelope and, at
// the end, the observable.
template <typename T, int MODE, int NS, bool HERM>
__device__ __forceinline__ void res_gwarp(const ResArgs& A, const ResGroup& g, unsigned char* sm, int gt, int gn, int bar) {
  using C = typename C2T<T>::type;
  const ResView<T, NS, HERM> V(A, g, sm, gt, gn, bar);
  constexpr int GW = V.GW;
  constexpr int GI = HERM ? 2 : 4;  // items per lane (M <= 64)
  const ResHdr& h = *reinterpret_cast<const ResHdr*>(V.blk);
  const ResWeights<T> W(V.blk, g.M);
  const int M = g.M, P = V.P, lane = gt & 31;
  const int nq = V.sep ? GW * M : 0;
  C* U = V.U;
  const C zero = cmk<C>(0.0, 0.0);

  C gy[GI], gs[GI], gc[GI], gd[GI];
  T gm[GI], gp[GI], rm[GI], rp[NS == 2 ? GI : 1];
  V.stage_in(V.yg, g.blk_elems);
#pragma unroll
  for (int i = 0; i < GI; ++i) {
    const int q = lane + 32 * i;
    gy[i] = gs[i] = gc[i] = gd[i] = zero;
    gm[i] = gp[i] = rm[i] = (T)0;
    if (NS == 2) rp[NS == 2 ? i : 0] = (T)0;
    if (q < nq) {
      const bool isx = q < M;
      const int k = isx ? q : q - M;
      gy[i] = U[isx ? k : g.gy_off + k];
      gd[i] = isx ? cadd(W.dx[k], cmk<C>(g.c_re, g.c_im)) : cadd(W.dy[k], cmk<C>(-g.c_re, -g.c_im));
      gm[i] = isx ? W.xm[k] : W.ym[k];
      gp[i] = isx ? W.xp[k] : W.yp[k];
      if (isx && k + 1 < M) rm[i] = W.smx[k + 1];
      if (NS == 2 && isx && k > 0) rp[NS == 2 ? i : 0] = W.spx[k - 1];
    }
  }
  V.sync();
  if (!A.comp_zero) {
    V.stage_in(V.cg, g.blk_elems);
#pragma unroll
    for (int i = 0; i < GI; ++i) {
      const int q = lane + 32 * i;
      if (q < nq) gc[i] = U[q < M ? q : g.gy_off + q - M];
    }
    V.sync();
  }
  // the envelope's 32 stages from step s0 on, one per lane, into half (s0 / 8) & 1 of the table
  auto envelope = [&](int s0) {
    const int step = s0 + (lane >> 2), stage = (lane & 3) + 1;
    C a = cmk<C>(h.a_re, h.a_im);
    if (h.ch) {
      const double tau = A.tau0 + (double)(A.step0 + step) * A.dt;
      const double t = pipe_chan_time(1, tau, stage, A.dt, A.horizon, A.reverse);
      const double tm = pipe_chan_time(2, tau, stage, A.dt, A.horizon, A.reverse);
      float t32[2];
      t32[0] = (float)t;
      t32[1] = (float)(t - (double)t32[0]);
      C e = pipe_chan_value<T>(h.chan, A.chpar, t, tm, t32);
      if (h.conj) e.y = -e.y;
      a = cmul(a, e);
    }
    V.E[((s0 >> 3) & 1) * 32 + lane] = a;
  };
  // stage input v of this lane's item i into half b: the value, and as row products
  auto put = [&](int b, int i, C v) {
    const int q = lane + 32 * i;
    V.Gs[b * GW * P + (q < M ? q : q - M + P)] = v;
    if (q < M) {
      C* r = V.RG + b * 4 * P;
      const C p = cscale(v, rm[i]);
      if (q + 1 < M) {
        r[q + 1] = p;
        if (HERM) r[P + q + 1] = p;
      }
      if constexpr (NS == 2) {
        const C p2 = cscale(v, rp[i]);
        if (q > 0) {
          r[2 * P + q - 1] = p2;
          if (HERM) r[3 * P + q - 1] = p2;
        }
      }
    }
  };
  for (int i = lane; i < 8 * P; i += 32) V.RG[i] = zero;
  for (int i = lane; i < 4 * P; i += 32) V.Gs[i] = zero;
  __syncwarp();
#pragma unroll
  for (int i = 0; i < GI; ++i)
    if (lane + 32 * i < nq) put(0, i, gy[i]);
  envelope(0);
  V.sync();

  const T hh = res_const<T>(A, 0), h2 = res_const<T>(A, 1), w_hi = res_const<T>(A, 2), w_lo = res_const<T>(A, 3);
  auto rhs = [&](int b, int i, C a) {
    const int q = lane + 32 * i;
    const bool isx = q < M;
    const int k = isx ? q : q - M;
    const C* G = V.Gs + b * GW * P + (isx ? 0 : P);
    const C lo = cscale(G[max(k - 1, 0)], gm[i]), hi = cscale(G[min(k + 1, M - 1)], gp[i]);
    // X: a lo - conj(a) hi;  Y: conj(a) lo - a hi
    return off_diag<MODE>(conj_if(a, isx ? 0u : 0x80000000u), lo, hi, cmul(gd[i], G[k]));
  };

  const int n_steps = A.n_steps;
#pragma unroll 1
  for (int step = 0; step < n_steps; ++step) {
    const C* Es = V.E + ((step >> 3) & 1) * 32 + (step & 7) * 4;
#pragma unroll 1
    for (int stage = 1; stage <= 3; ++stage) {
      const int b = (stage & 1) ^ 1;
      const C a = Es[stage - 1];
      const T al = stage == 3 ? hh : h2, be = stage == 1 ? (T)1 : (T)2;
#pragma unroll
      for (int i = 0; i < GI; ++i) {
        if (lane + 32 * i >= nq) continue;
        const C k = rhs(b, i, a);
        gs[i] = caxpy(be, k, gs[i]);
        put(b ^ 1, i, caxpy(al, k, gy[i]));
      }
      if (stage == 1 && (step & 7) == 4 && (step | 7) + 1 < n_steps) envelope((step | 7) + 1);
      V.sync();
    }
    const C a = Es[3];
#pragma unroll
    for (int i = 0; i < GI; ++i) {
      if (lane + 32 * i >= nq) continue;
      const C k = rhs(1, i, a);
      C d;
      d.x = fma(w_hi, gs[i].x + k.x, fma(w_lo, gs[i].x + k.x, -gc[i].x));
      d.y = fma(w_hi, gs[i].y + k.y, fma(w_lo, gs[i].y + k.y, -gc[i].y));
      res_update(d, gy[i], gc[i]);
      gs[i] = zero;
      put(0, i, gy[i]);
    }
    V.sync();
  }

  V.sync();
  auto place = [&](const C (&v)[GI]) {
#pragma unroll
    for (int i = 0; i < GI; ++i) {
      const int q = lane + 32 * i;
      if (q >= nq) continue;
      U[q < M ? q : g.gy_off + q - M] = v[i];
      if (HERM) U[g.gy_off + q] = conj_if(v[i], 0x80000000u);
    }
    // the padding of the blocks stays zero
    if (V.sep)
      for (int i = M + lane; i < g.gy_off; i += 32) {
        U[i] = zero;
        U[g.gy_off + i] = zero;
      }
    for (int i = g.r_off + M * M + lane; i < g.blk_elems; i += 32) U[i] = zero;
  };
  place(gy);
  V.stage_out(V.yg, g.blk_elems);
  place(gc);
  V.stage_out(V.cg, g.blk_elems);
  // Tr(rho0 A)'s contribution: w sum_e f_e (G_x[k] G_y[l] + R[k, l]) of y - comp
  const PipeObs<double2>* ob = reinterpret_cast<const PipeObs<double2>*>(V.blk + h.obs_off);
  double2 v = make_double2(0.0, 0.0);
  auto val = [&](int i) {
    const C p = V.yg[i], q = V.cg[i];
    return make_double2((double)(p.x - q.x), (double)(p.y - q.y));
  };
  if (lane < h.n_obs) {
    const PipeObs<double2> o = ob[lane];
    v = val(g.r_off + o.kx * M + o.ly);
    if (V.sep) v = cadd(v, cmul(val(o.kx), val(g.gy_off + o.ly)));
    v = cmul(cmul(make_double2(g.w_re, g.w_im), o.f), v);
  }
  if (h.n_obs > 1) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      v.x += __shfl_down_sync(0xffffffffu, v.x, o);
      v.y += __shfl_down_sync(0xffffffffu, v.y, o);
    }
  }
  if (lane == 0) A.obs[g.sys] = v;
}

template <typename T, int MODE, int NS, bool SD, bool HERM>
__global__ void __launch_bounds__(32 * BQ_RES_WARPS(2 * sizeof(T), HERM), sizeof(T) == 4 ? 2 : 1)
    k_resident(const ResArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5;
  const int gi = A.bins[blockIdx.x].g[warp];
  if (gi < 0) return;
  const ResGroup g = A.groups[gi];
  if (A.flags && (A.flags[g.sys] != 0) != (A.want != 0)) return;
  const int gt = (int)threadIdx.x - 32 * g.warp0, gn = 32 * g.nwarps;
  {  // The residual and the parameters are read after the state, each behind a barrier: ask for them now.
     // (One step of 65 536 systems, whose arrays come from HBM: 1394 -> 1313 us, the streamed step
     // kernel 1331; 16 384: 358 -> 337; 4096, all in L2: 79 -> 80.)
    const int eb = 2 * sizeof(T), nc = A.comp_zero ? 0 : g.blk_elems * eb;
    const char* c = reinterpret_cast<const char*>(A.comp) + (size_t)g.blk_off * eb;
    for (int o = gt * 128; o < nc; o += gn * 128) prefetch_l2(c + o);
    const char* b = reinterpret_cast<const char*>(A.params) + g.param_off;
    const int nb = (int)sizeof(ResHdr) + g.M * (2 * eb + 8 * (int)sizeof(T));
    for (int o = gt * 128; o < nb; o += gn * 128) prefetch_l2(b + o);
  }
  const int bar = 1 + g.warp0 / 2;  // groups have at least two warps
  unsigned char* sm = smem_raw + g.smem_off;
  if (gt >= gn - 32) {
    res_gwarp<T, MODE, NS, HERM>(A, g, sm, gt, gn, bar);
    return;
  }
  // (the strip lengths res_shape chooses from)
  if constexpr (sizeof(T) == 8) {
    if (g.rb == 2) res_strips<T, 2, MODE, NS, SD, HERM>(A, g, sm, gt, gn, bar);
    else res_strips<T, 4, MODE, NS, SD, HERM>(A, g, sm, gt, gn, bar);
  } else if constexpr (HERM) {
    if (g.rb == 3) res_strips<T, 3, MODE, NS, SD, HERM>(A, g, sm, gt, gn, bar);
    else res_strips<T, 5, MODE, NS, SD, HERM>(A, g, sm, gt, gn, bar);
  } else {
    switch (g.rb) {
      case 2: res_strips<T, 2, MODE, NS, SD, HERM>(A, g, sm, gt, gn, bar); break;
      case 4: res_strips<T, 4, MODE, NS, SD, HERM>(A, g, sm, gt, gn, bar); break;
      default: res_strips<T, 7, MODE, NS, SD, HERM>(A, g, sm, gt, gn, bar); break;
    }
  }
}

template <typename T, int MODE, int NS, bool SD, bool HERM>
static cudaError_t launch_resident_one(const ResArgs& a, int n_bins, int smem_bytes, cudaStream_t s) {
  // (per call: the attribute belongs to the current device's context, and setting it is cheap)
  cudaError_t e = cudaFuncSetAttribute(k_resident<T, MODE, NS, SD, HERM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       BQ_RES_SMEM_MAX);
  if (e != cudaSuccess) return e;
  k_resident<T, MODE, NS, SD, HERM><<<n_bins, 32 * BQ_RES_WARPS(2 * sizeof(T), HERM), smem_bytes, s>>>(a);
  return cudaGetLastError();
}

// variant: bit 0 = a general off-diagonal coefficient, bit 1 = a sandwich term with source (k + 1, l + 1),
// bit 2 = sandwich terms restricted to k = l
template <typename T, bool HERM>
static cudaError_t launch_resident_t(const ResArgs& a, int variant, int n_bins, int smem_bytes, cudaStream_t s) {
  if (n_bins <= 0) return cudaSuccess;
  switch (variant) {
    case 0: return launch_resident_one<T, 1, 1, false, HERM>(a, n_bins, smem_bytes, s);
    case 1: return launch_resident_one<T, 2, 1, false, HERM>(a, n_bins, smem_bytes, s);
    case 2: return launch_resident_one<T, 1, 2, false, HERM>(a, n_bins, smem_bytes, s);
    case 3: return launch_resident_one<T, 2, 2, false, HERM>(a, n_bins, smem_bytes, s);
    case 4: return launch_resident_one<T, 1, 1, true, HERM>(a, n_bins, smem_bytes, s);
    case 5: return launch_resident_one<T, 2, 1, true, HERM>(a, n_bins, smem_bytes, s);
    case 6: return launch_resident_one<T, 1, 2, true, HERM>(a, n_bins, smem_bytes, s);
    default: return launch_resident_one<T, 2, 2, true, HERM>(a, n_bins, smem_bytes, s);
  }
}

}  // namespace bq
