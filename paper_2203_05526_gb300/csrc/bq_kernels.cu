// CUDA kernels of the mapped adjoint-Lindblad solver (sm_103a).
//
//  * k_stage     one fused classical-RK4 stage of the coupled system of Eqs. 9a-c / 303a-c
//                (or of Eq. 3 itself for the direct number-basis method): stencil terms of
//                H and of the dissipators, the separable source S(G_x G_y), and the RK4
//                combine, for every point of a tile staged in shared memory.
//  * k_eval      observables of Eqs. 7 / 11: warp reductions over initial conditions.
//  * k_scatter   initial state (Eqs. 10, 13).
//
// Memory-bound by design: the stencil has reach one per variable and ~8-12 complex terms
// per point, so it never touches the tensor cores.  Loads of the stage input are staged
// once per CTA in shared memory (halo re-reads come from there), the state, stage output
// and accumulator are streamed with coalesced accesses.
#include <type_traits>
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "bq_device.cuh"
#include "bq_internal.h"
#include "bq_launch.h"

namespace bq {

// ---------------------------------------------------------------------------------------
// Drive envelopes (channel kinds of bq.h).
// ---------------------------------------------------------------------------------------
__device__ double2 chan_value(const ChanDesc& c, const double* par, double t) {
  const double* p = par + c.par_off;
  switch (c.kind) {
    case 0:  // CONST
      return make_double2(p[0], p[1]);
    case 1: {  // GAUSS
      const double d = t - p[2];
      const double e = exp(-(d * d) / (2.0 * p[3] * p[3]));
      return make_double2(p[0] * e, p[1] * e);
    }
    case 2: {  // PWC
      const int n_seg = (c.n_par - 2) / 2;
      const double x = floor((t - p[0]) / p[1]);
      if (!(x >= 0.0) || x >= (double)n_seg) return make_double2(0.0, 0.0);
      const int s = (int)x;
      return make_double2(p[2 + 2 * s], p[3 + 2 * s]);
    }
    case 3: {  // CEXP
      double sn, cs;
      sincos(p[2] * t, &sn, &cs);
      return make_double2(p[0] * cs - p[1] * sn, p[0] * sn + p[1] * cs);
    }
    default:
      return make_double2(0.0, 0.0);
  }
}

// Coefficient of term t at the current stage: c * [channel or its conjugate].
__device__ __forceinline__ double2 term_coef(const TermDesc& td, const ChanDesc* chans, const double* chpar,
                                             double tau_step, double dt, int stage, double horizon, int reverse) {
  double2 c = make_double2(td.c_re, td.c_im);
  if (td.ch >= 0) {
    const ChanDesc cd = chans[td.ch];
    const double tau = (cd.kind == 2) ? tau_step + 0.5 * dt : tau_step + stage_c(stage) * dt;
    const double t = reverse ? horizon - tau : tau;
    double2 e = chan_value(cd, chpar, t);
    if (td.conj) e.y = -e.y;
    c = make_double2(c.x * e.x - c.y * e.y, c.x * e.y + c.y * e.x);
  }
  return c;
}

// ---------------------------------------------------------------------------------------
// Fused RK4 stage.
// ---------------------------------------------------------------------------------------
// One work item of a stage (k_stage: one item per CTA; the cooperative segment kernels: the
// CTA's items of every stage of a segment).  tau: tau at the start of the step.  fresh: load
// the item's descriptors (else the shared-memory copies of the CTA's previous call, for the
// same item, are reused and only the stage coefficients are re-evaluated).
template <typename T, int NM>
__device__ __forceinline__ void stage_body(const StageArgs& A, int item, double tau, bool fresh) {
  using C = typename C2T<T>::type;
  constexpr int ND = 2 * NM;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* win = reinterpret_cast<C*>(smem_raw);

  __shared__ SysDesc sd;
  __shared__ WorkItem wi;
  __shared__ TermDesc st[BQ_MAX_TERMS];
  __shared__ C sc[BQ_MAX_TERMS];
  __shared__ int cwoff[BQ_MAX_TERMS];
  __shared__ double s_tau;

  const int tid = threadIdx.x;
  __syncthreads();  // the CTA's previous item is done with the shared copies
  if (tid == 0) {
    if (fresh) {
      wi = A.work[item];
      sd = A.sys[wi.sys];
    }
    s_tau = tau;
  }
  __syncthreads();
  const int nt = sd.n_terms;
  for (int t = tid; t < nt; t += blockDim.x) {
    if (fresh) st[t] = A.terms[sd.term_off + t];
    const double2 c = term_coef(st[t], A.chans, A.chpar, s_tau, A.dt, A.stage, A.horizon, A.reverse);
    sc[t] = cmk<C>(c.x, c.y);
  }
  if (fresh && tid == 32) {  // offsets of the coefficient x weight tables (one table per term)
    int o = 0;
    for (int t = 0; t < nt; ++t) {
      const TermDesc& td = A.terms[sd.term_off + t];
      cwoff[t] = o;
      o += td.n_act > 0 ? sd.M[td.dim[0] % NM] : 1;
    }
  }
  // Stage the R window and (for the separable part) G_x, G_y of the stage input.
  const C* uin = reinterpret_cast<const C*>(A.u_in);
  const int wn = wi.win_hi - wi.win_lo;
  if (sd.has_r && !wi.gread) {
    const C* src = uin + sd.off_r + wi.win_lo;
    for (int i = tid; i < wn; i += blockDim.x) win[i] = src[i];
  }
  // R source at flat index i of the system: the staged window, or global memory for tiles
  // whose halo does not fit in shared memory
  const C* urg = uin + (sd.has_r ? sd.off_r : 0);
  auto rsrc_at = [&](int i) { return wi.gread ? urg[i] : win[i - wi.win_lo]; };
  C* gxs = win + wn;
  C* gys = gxs + sd.n_g;
  const bool do_sep = sd.has_sep && wi.sep_hi > wi.sep_lo;
  if (sd.has_sep && (do_sep || sd.has_r)) {
    const C* sx = uin + sd.off_gx;
    const C* sy = uin + sd.off_gy;
    for (int i = tid; i < sd.n_g; i += blockDim.x) {
      gxs[i] = sx[i];
      gys[i] = sy[i];
    }
  }
  __syncthreads();

  const T* W = reinterpret_cast<const T*>(A.wtab);
  // Coefficient x weight tables: cw_t[i] = c_t(stage) W_t,0[i] over the index of the term's
  // first active dimension, so that a point's term costs one complex multiply-add (times the
  // weights of further active dimensions) instead of weight products and a scaling.
  C* cw = win + wn + (sd.has_sep ? 2 * sd.n_g : 0);
  {
    const int nwarp = (int)blockDim.x >> 5, lane = tid & 31;
    for (int t = tid >> 5; t < nt; t += nwarp) {
      const TermDesc& td = st[t];
      if (td.n_act == 0) {
        if (lane == 0) cw[cwoff[t]] = sc[t];
      } else {
        const int len = sd.M[td.dim[0] % NM];
        for (int i = lane; i < len; i += 32) cw[cwoff[t] + i] = cscale(sc[t], W[td.wtab[0] + i]);
      }
    }
  }
  __syncthreads();
  const C* D = reinterpret_cast<const C*>(A.diag) + sd.diag_off;
  C* uout = reinterpret_cast<C*>(A.u_out);
  C* y = reinterpret_cast<C*>(A.y);
  C* acc = reinterpret_cast<C*>(A.acc);
  const T dt = (T)A.dt;
  const int stage = A.stage;
  int Md[ND];
#pragma unroll
  for (int d = 0; d < ND; ++d) Md[d] = sd.M[d % NM];
  // diag table offsets: dim d's table starts at sum_{d' < d} M_d'
  int doff[ND];
  {
    int o = 0;
#pragma unroll
    for (int d = 0; d < ND; ++d) { doff[d] = o; o += Md[d]; }
  }

  // Classical RK4 with the stage sum kept as an increment (inc = k1 + 2 k2 + 2 k3) and a
  // compensated (Kahan) update of the state at stage 4, y += dt/6 (inc + k4): in FP32 the
  // per-step increment is a few ulps of y, and adding partial increments to y four times
  // per step (or even once without compensation) biases the rounding in one direction.
  C* comp = reinterpret_cast<C*>(A.comp);
  auto combine = [&](int64_t gi, C uc, C k) {
    if (stage == 1) {
      uout[gi] = caxpy(dt * (T)0.5, k, uc);
      acc[gi] = k;
    } else if (stage == 4) {
      const C yv = y[gi];
      const C s = cadd(acc[gi], k);
      const C cv = comp[gi];
      C d, t, c2;
      d.x = dt * (T)(1.0 / 6.0) * s.x - cv.x;
      d.y = dt * (T)(1.0 / 6.0) * s.y - cv.y;
      t.x = yv.x + d.x;
      t.y = yv.y + d.y;
      c2.x = (t.x - yv.x) - d.x;
      c2.y = (t.y - yv.y) - d.y;
      y[gi] = t;
      comp[gi] = c2;
    } else {
      const C yv = y[gi];
      uout[gi] = caxpy(stage == 2 ? dt * (T)0.5 : dt, k, yv);
      acc[gi] = caxpy((T)2, k, acc[gi]);
    }
  };

  // Each point is handled by a group of L = A.lanes adjacent lanes: lane `sub` of the group
  // sums the terms t = sub, sub + L, ... (the first lane also the diagonal part), the group
  // combines its partial sums with shuffles and the first lane writes the point.  L = 1
  // keeps the plain one-thread-per-point loop; L > 1 gives the small launches of a few large
  // systems more warps to hide latency with.
  const int L = A.lanes;
  const int sub = tid & (L - 1);
  const unsigned gmask = L == 1 ? (1u << (tid & 31)) : (((1u << L) - 1u) << ((tid & 31) & ~(L - 1)));
  const int pstride = (int)blockDim.x / L;
  auto group_sum = [&](C k) {
    for (int o = 1; o < L; o <<= 1) {
      k.x += __shfl_xor_sync(gmask, k.x, o);
      k.y += __shfl_xor_sync(gmask, k.y, o);
    }
    return k;
  };

  // ---- R points of the tile -------------------------------------------------------
  if (sd.has_r) {
    const int ng = sd.n_g;
    for (int p = wi.start + tid / L; p < wi.start + wi.len; p += pstride) {
      int idx[ND];
      const int kx = sd.r_diag ? p : p / ng;  // diagonal residual layout: point p is (p, p)
      const int ly = sd.r_diag ? p : p - kx * ng;
      {
        int r = kx;
#pragma unroll
        for (int d = NM - 1; d >= 0; --d) { idx[d] = r % Md[d]; r /= Md[d]; }
        r = ly;
#pragma unroll
        for (int d = ND - 1; d >= NM; --d) { idx[d] = r % Md[d]; r /= Md[d]; }
      }
      const C uc = rsrc_at(p);
      C k = cmk<C>(0.0, 0.0);
      if (sub == 0) {
        C dg = D[doff[0] + idx[0]];
#pragma unroll
        for (int d = 1; d < ND; ++d) dg = cadd(dg, D[doff[d] + idx[d]]);
        k = cmul(dg, uc);
      }
      for (int t = sub; t < nt; t += L) {
        const TermDesc& td = st[t];
        if (td.diagp1 && idx[td.diagp1 - 1] != idx[NM + td.diagp1 - 1]) continue;  // projector P
        // coefficient x weights; the source is inside the grid exactly when every shifted
        // index is (else every weight table holds a zero at this point)
        C c = cw[cwoff[t] + (td.n_act > 0 ? idx[td.dim[0]] : 0)];
        bool in = true;
        for (int i = 0; i < td.n_act; ++i) {
          const int d = td.dim[i];
          in = in && (unsigned)(idx[d] + td.sh[i]) < (unsigned)Md[d];
          if (i > 0) c = cscale(c, W[td.wtab[i] + idx[d]]);
        }
        // diagonal layout: only terms that shift x and y alike have an R source, at deltaGx
        const bool rsrc = !sd.r_diag || td.deltaGx == td.deltaGy;
        C v;
        if (td.side == SIDE_S && sd.has_sep) {
          // c (R[src] + G_x[kx + sx] G_y[ly + sy])
          v = in ? cmul(gxs[kx + td.deltaGx], gys[ly + td.deltaGy]) : cmk<C>(0.0, 0.0);
          if (rsrc && in) v = cadd(rsrc_at(p + (sd.r_diag ? td.deltaGx : td.deltaR)), v);
        } else {
          if (!rsrc || !in) continue;
          v = rsrc_at(p + (sd.r_diag ? td.deltaGx : td.deltaR));
        }
        k = cfma(c, v, k);
      }
      k = group_sum(k);
      if (sub == 0) {
        if (A.rec) reinterpret_cast<C*>(A.rec)[sd.off_r + p] = uc;
        combine(sd.off_r + p, uc, k);
      }
    }
  }

  // ---- separable part: G_x (left operator + C) and G_y (right operator - C) --------
  if (do_sep) {
    const C Cc = cmk<C>(sd.c_re, sd.c_im);
    const int ng = sd.n_g;
    for (int i = wi.sep_lo + tid / L; i < wi.sep_hi; i += pstride) {
      const int side = i < ng ? SIDE_X : SIDE_Y;
      const int g = side == SIDE_X ? i : i - ng;
      const int d0 = side == SIDE_X ? 0 : NM;
      int idx[ND];
      {
        int r = g;
#pragma unroll
        for (int d = NM - 1; d >= 0; --d) { idx[d0 + d] = r % Md[d]; r /= Md[d]; }
      }
      const C* gs = side == SIDE_X ? gxs : gys;
      const C uc = gs[g];
      C k = cmk<C>(0.0, 0.0);
      if (sub == 0) {
        C dg = side == SIDE_X ? Cc : cmk<C>(-sd.c_re, -sd.c_im);
#pragma unroll
        for (int d = 0; d < NM; ++d) dg = cadd(dg, D[doff[d0 + d] + idx[d0 + d]]);
        k = cmul(dg, uc);
      }
      for (int t = sub; t < nt; t += L) {
        const TermDesc& td = st[t];
        if (td.side != side) continue;
        C c = cw[cwoff[t] + (td.n_act > 0 ? idx[td.dim[0]] : 0)];
        bool in = true;
        for (int j = 0; j < td.n_act; ++j) {
          const int d = td.dim[j];
          in = in && (unsigned)(idx[d] + td.sh[j]) < (unsigned)Md[d];
          if (j > 0) c = cscale(c, W[td.wtab[j] + idx[d]]);
        }
        if (!in) continue;
        k = cfma(c, gs[g + (side == SIDE_X ? td.deltaGx : td.deltaGy)], k);
      }
      k = group_sum(k);
      if (sub == 0) {
        if (A.rec) reinterpret_cast<C*>(A.rec)[(side == SIDE_X ? sd.off_gx : sd.off_gy) + g] = uc;
        combine((side == SIDE_X ? sd.off_gx : sd.off_gy) + g, uc, k);
      }
    }
  }

}

template <typename T, int NM>
__global__ void __launch_bounds__(BQ_BLOCK) k_stage(const StageArgs A) {
  stage_body<T, NM>(A, blockIdx.x, A.tau_base[0] + (double)(*(volatile long long*)A.counter) * A.dt, true);
  // ---- step bookkeeping: the last CTA of stage 4 advances the step counter ----------
  if (A.stage == 4) {
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      const unsigned int t = atomicAdd(A.ticket, 1u);
      if (t == gridDim.x - 1) {
        *A.ticket = 0u;
        *A.counter = *(volatile long long*)A.counter + 1;
        __threadfence();
      }
    }
  }
}

// ---------------------------------------------------------------------------------------
// Fused RK4 stage, single-mode fast path (the batched workloads of the paper's oscillator
// family).  One CTA holds one whole system: R (M x M), G_x, G_y, the diagonal tables and the
// weight tables of its few stencil terms, all in shared memory.  The term program (counts,
// shifts, table offsets) is precompiled on the host into one M1Sys record per system, read
// with one coalesced load, so a CTA has exactly two barriers.  Per point:
//   k(k,l) = (D_x[k] + D_y[l]) u[k,l] + sum_X c W[k] u[k+s,l] + sum_Y c W[l] u[k,l+s]
//          + sum_S c Wx[k] Wy[l] (u[k+sx,l+sy] + G_x[k+sx] G_y[l+sy]).
// Out-of-grid sources have zero weight; their (clamped) address stays inside the tile.
// ---------------------------------------------------------------------------------------
// Envelope value in the state's precision (FP32 envelopes are accurate to ~1e-7 relative,
// far inside the FP32 path's tolerance; FP64 states evaluate in FP64).
template <typename T>
__device__ double2 chan_value_t(const ChanDesc& c, const double* p, double t) {
  p += c.par_off;
  if (c.kind == 1) {
    const T d = (T)(t - p[2]);
    const T e = dev_exp<T>(-(d * d) / ((T)2 * (T)p[3] * (T)p[3]));
    return make_double2(p[0] * (double)e, p[1] * (double)e);
  }
  return chan_value(c, p - c.par_off, t);
}

template <typename T, int MX, int MY, int MS>
__global__ void __launch_bounds__(BQ_BLOCK) k_stage_m1(const StageArgs A, const M1Sys* __restrict__ m1) {
  using C = typename C2T<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ M1Sys s;
  __shared__ C coef[3 * BQ_M1_MAXT];
  __shared__ double s_tau;
  const int tid = threadIdx.x;
  {
    const int* src = reinterpret_cast<const int*>(m1 + blockIdx.x);
    int* dst = reinterpret_cast<int*>(&s);
    for (int i = tid; i < (int)(sizeof(M1Sys) / sizeof(int)); i += blockDim.x) dst[i] = src[i];
    if (tid == 0) s_tau = A.tau_base[0] + (double)(*(volatile long long*)A.counter) * A.dt;
  }
  __syncthreads();
  const int M = s.M, nX = s.nX, nY = s.nY, nS = s.nS;
  const int sdiag = s.sdiag;  // bit q: sandwich term q acts only where k = l
  const int has_r = s.has_r, has_sep = s.has_sep;
  const int nr = has_r ? M * M : 0;
  // shared layout: u[M*M] | gx[M] | gy[M] | dx[M] | dy[M] | wX[nX*M] wY[nY*M] wSx[nS*M] wSy[nS*M] (real)
  C* u = reinterpret_cast<C*>(smem_raw);
  C* gx = u + nr;
  C* gy = gx + M;
  C* dx = gy + M;
  C* dy = dx + M;
  T* wt = reinterpret_cast<T*>(dy + M);
  T* wX = wt;
  T* wY = wX + nX * M;
  T* wSx = wY + nY * M;
  T* wSy = wSx + nS * M;
  // term coefficients at this stage's time (one thread per term)
  {
    const int nt = nX + nY + nS;
    if (tid < nt) {
      const int t = tid < nX ? s.tX[tid] : (tid < nX + nY ? s.tY[tid - nX] : s.tS[tid - nX - nY]);
      const TermDesc& td = A.terms[s.term_off + t];
      double2 c = make_double2(td.c_re, td.c_im);
      if (td.ch >= 0) {
        const ChanDesc cd = A.chans[td.ch];
        const double tau = (cd.kind == 2) ? s_tau + 0.5 * A.dt : s_tau + stage_c(A.stage) * A.dt;
        double2 e = chan_value_t<T>(cd, A.chpar, A.reverse ? A.horizon - tau : tau);
        if (td.conj) e.y = -e.y;
        c = make_double2(c.x * e.x - c.y * e.y, c.x * e.y + c.y * e.x);
      }
      coef[tid] = cmk<C>(c.x, c.y);
    }
  }
  const C* uin = reinterpret_cast<const C*>(A.u_in);
  if (has_r) {
    const C* src = uin + s.off_r;
    for (int i = tid; i < nr; i += blockDim.x) u[i] = src[i];
  }
  if (has_sep)
    for (int i = tid; i < M; i += blockDim.x) {
      gx[i] = uin[s.off_gx + i];
      gy[i] = uin[s.off_gy + i];
    }
  {
    const C* Dg = reinterpret_cast<const C*>(A.diag) + s.diag_off;
    const T* W = reinterpret_cast<const T*>(A.wtab);
    for (int i = tid; i < M; i += blockDim.x) {
      dx[i] = Dg[i];
      dy[i] = Dg[M + i];
#pragma unroll
      for (int j = 0; j < MX; ++j) if (j < nX) wX[j * M + i] = s.wX[j] >= 0 ? W[s.wX[j] + i] : (T)1;
#pragma unroll
      for (int j = 0; j < MY; ++j) if (j < nY) wY[j * M + i] = s.wY[j] >= 0 ? W[s.wY[j] + i] : (T)1;
#pragma unroll
      for (int j = 0; j < MS; ++j)
        if (j < nS) {
          wSx[j * M + i] = s.wSx[j] >= 0 ? W[s.wSx[j] + i] : (T)1;
          wSy[j * M + i] = s.wSy[j] >= 0 ? W[s.wSy[j] + i] : (T)1;
        }
    }
  }
  __syncthreads();

  C cX[MX], cY[MY], cS[MS];
  int shX[MX], shY[MY], shSx[MS], shSy[MS];
#pragma unroll
  for (int j = 0; j < MX; ++j) { cX[j] = coef[min(j, 3 * BQ_M1_MAXT - 1)]; shX[j] = s.sX[j]; }
#pragma unroll
  for (int j = 0; j < MY; ++j) { cY[j] = coef[min(nX + j, 3 * BQ_M1_MAXT - 1)]; shY[j] = s.sY[j]; }
#pragma unroll
  for (int j = 0; j < MS; ++j) { cS[j] = coef[min(nX + nY + j, 3 * BQ_M1_MAXT - 1)]; shSx[j] = s.sSx[j]; shSy[j] = s.sSy[j]; }

  C* uout = reinterpret_cast<C*>(A.u_out);
  C* y = reinterpret_cast<C*>(A.y);
  C* acc = reinterpret_cast<C*>(A.acc);
  C* comp = reinterpret_cast<C*>(A.comp);
  const T dt = (T)A.dt;
  const int stage = A.stage;
  auto combine = [&](int64_t gi, C uc, C kv) {
    if (stage == 1) {
      uout[gi] = caxpy(dt * (T)0.5, kv, uc);
      acc[gi] = kv;
    } else if (stage == 4) {
      const C yv = y[gi];
      const C sm = cadd(acc[gi], kv);
      const C cv = comp[gi];
      C d, t, c2;
      d.x = dt * (T)(1.0 / 6.0) * sm.x - cv.x;
      d.y = dt * (T)(1.0 / 6.0) * sm.y - cv.y;
      t.x = yv.x + d.x;
      t.y = yv.y + d.y;
      c2.x = (t.x - yv.x) - d.x;
      c2.y = (t.y - yv.y) - d.y;
      y[gi] = t;
      comp[gi] = c2;
    } else {
      const C yv = y[gi];
      uout[gi] = caxpy(stage == 2 ? dt * (T)0.5 : dt, kv, yv);
      acc[gi] = caxpy((T)2, kv, acc[gi]);
    }
  };

  if (has_r) {
    const float invM = 1.0f / (float)M;
    for (int p = tid; p < nr; p += blockDim.x) {
      const int kx = (int)(((float)p + 0.5f) * invM);
      const int ly = p - kx * M;
      const C uc = u[p];
      C kv = cmul(cadd(dx[kx], dy[ly]), uc);
#pragma unroll
      for (int j = 0; j < MX; ++j)
        if (j < nX) {
          const int r = min(max(kx + shX[j], 0), M - 1);
          kv = cfma(cX[j], cscale(u[r * M + ly], wX[j * M + kx]), kv);
        }
#pragma unroll
      for (int j = 0; j < MY; ++j)
        if (j < nY) {
          const int c = min(max(ly + shY[j], 0), M - 1);
          kv = cfma(cY[j], cscale(u[kx * M + c], wY[j * M + ly]), kv);
        }
#pragma unroll
      for (int j = 0; j < MS; ++j)
        if (j < nS && (!((sdiag >> j) & 1) || kx == ly)) {  // secular projector: k = l only
          const int r = min(max(kx + shSx[j], 0), M - 1);
          const int c = min(max(ly + shSy[j], 0), M - 1);
          C v = u[r * M + c];
          if (has_sep) v = cadd(v, cmul(gx[r], gy[c]));
          kv = cfma(cS[j], cscale(v, wSx[j * M + kx] * wSy[j * M + ly]), kv);
        }
      if (A.rec) reinterpret_cast<C*>(A.rec)[s.off_r + p] = uc;
      combine(s.off_r + p, uc, kv);
    }
  }
  if (has_sep) {
    for (int i = tid; i < 2 * M; i += blockDim.x) {
      const bool isx = i < M;
      const int g = isx ? i : i - M;
      const C* gs = isx ? gx : gy;
      C dg = isx ? cadd(dx[g], cmk<C>(s.c_re, s.c_im)) : cadd(dy[g], cmk<C>(-s.c_re, -s.c_im));
      C kv = cmul(dg, gs[g]);
      if (isx) {
#pragma unroll
        for (int j = 0; j < MX; ++j)
          if (j < nX) kv = cfma(cX[j], cscale(gs[min(max(g + shX[j], 0), M - 1)], wX[j * M + g]), kv);
      } else {
#pragma unroll
        for (int j = 0; j < MY; ++j)
          if (j < nY) kv = cfma(cY[j], cscale(gs[min(max(g + shY[j], 0), M - 1)], wY[j * M + g]), kv);
      }
      if (A.rec) reinterpret_cast<C*>(A.rec)[(isx ? s.off_gx : s.off_gy) + g] = gs[g];
      combine((isx ? s.off_gx : s.off_gy) + g, gs[g], kv);
    }
  }
  if (stage == 4) {
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      const unsigned int t = atomicAdd(A.ticket, 1u);
      if (t == gridDim.x - 1) {
        *A.ticket = 0u;
        *A.counter = *(volatile long long*)A.counter + 1;
        __threadfence();
      }
    }
  }
}

// ---------------------------------------------------------------------------------------
// Pipelined single-mode stage (the HBM-streaming form of the fused stage).
//
// A persistent CTA processes its systems in order; thread 0 keeps n_slots - 1 systems in
// flight by issuing 1-D bulk copies (TMA, cp.async.bulk with an mbarrier transaction count)
// of each system's parameter block, stage coefficients, stage input, state, stage sum and
// compensation into a shared-memory slot, while all threads compute the current system from
// shared memory and stream the results to HBM with coalesced stores.  Every wait on an
// mbarrier is bounded; a wait that gives up sets an error word and the CTA returns.
// ---------------------------------------------------------------------------------------
// Element (1 + sx, 1 + sy) of a 3x3 register window, selected without taking addresses (so
// the window stays in registers).
template <typename C>
__device__ __forceinline__ C pick9(const C (&w0)[3], const C (&w1)[3], const C (&w2)[3], int sx, int sy) {
  const C a = sy < 0 ? w0[0] : (sy > 0 ? w0[2] : w0[1]);
  const C b = sy < 0 ? w1[0] : (sy > 0 ? w1[2] : w1[1]);
  const C c = sy < 0 ? w2[0] : (sy > 0 ? w2[2] : w2[1]);
  return sx < 0 ? a : (sx > 0 ? c : b);
}

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
  unsigned done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return done != 0;
}
// try_wait with a suspend-time hint (ns): the thread sleeps until the phase completes or the
// hint elapses instead of spinning through short polls
__device__ __forceinline__ bool mbar_try_wait_for(unsigned long long* bar, unsigned parity, unsigned ns) {
  unsigned done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity), "r"(ns)
      : "memory");
  return done != 0;
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
// L2 prefetch of a contiguous global range (16-byte aligned start, size a multiple of 16)
__device__ __forceinline__ void bulk_prefetch_l2(const void* src, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
// Asynchronous copy of one complex value (8 or 16 bytes, naturally aligned) from global to
// shared memory; the issuing thread reads it after cp_async_wait_all.
template <typename C>
__device__ __forceinline__ void cp_async_c(C* dst, const C* src) {
  static_assert(sizeof(C) == 8 || sizeof(C) == 16, "complex FP32 or FP64");
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(dst)), "l"(src), "n"((int)sizeof(C))
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

#define BQ_PIPE_RB 16  // system records per batch (power of two)
#define BQ_WAIT_LIMIT (1 << 22)
#define BQ_WAIT_SUSPENDS (1 << 16)  // suspended polls of at most BQ_WAIT_HINT_NS each (< 1 s in all)
#define BQ_WAIT_HINT_NS 10000u

// Two adjacent complex values from a 16-byte aligned shared-memory address.
template <typename C>
__device__ __forceinline__ void ld_pair(const C* p, C& a, C& b);
template <>
__device__ __forceinline__ void ld_pair<float2>(const float2* p, float2& a, float2& b) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  a = make_float2(v.x, v.y);
  b = make_float2(v.z, v.w);
}
template <>
__device__ __forceinline__ void ld_pair<double2>(const double2* p, double2& a, double2& b) {
  a = p[0];
  b = p[1];
}
template <typename C>
__device__ __forceinline__ void st_pair(C* p, C a, C b);
template <>
__device__ __forceinline__ void st_pair<float2>(float2* p, float2 a, float2 b) {
  *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
}
template <>
__device__ __forceinline__ void st_pair<double2>(double2* p, double2 a, double2 b) {
  p[0] = a;
  p[1] = b;
}

// RK4 update of one element in the pipelined stage kernel.  The state value of an element is
// y - comp, with comp the (negated) rounding residual of the last update: the state advances
// by the classical RK4 increment accumulated in a stage sum s at the increment's own
// magnitude and added to y once per step with an error-free sum.  With h = dt:
//   stage 1: k1 = f(y); u_2 = y + h/2 k1; s = r + h/6 k1 with r = -comp the carried residual;
//   stage 2: k2 = f(u_2); y is recovered from the stored u_2 and s as u_2 - 3 s (up to r, a
//            few ulps: it only forms the next stage input); u_3 = y + h/2 k2, s += h/6 (2 k2);
//   stage 3: k3 = f(u_3); u_4 = y + h k3, s += h/6 (2 k3);
//   stage 4: k4 = f(u_4); p = s + h/6 k4; y + p = y' + e exactly (TwoSum); y = y', comp = -e.
// The weight h/6 is applied as an unevaluated sum w_hi + w_lo (w_hi = fl(h/6)): the four
// stages' weights then add up to h to far below the state's rounding, so the effective step
// does not drift from h over long horizons (a plain fl(h/6) is off by up to 3e-8 relative,
// a phase error of that size times the rotation angle).  Arrays moved per step and point:
// stage 1 y (stage input), comp in and u, s out; stage 2 u, s in and u, s out; stage 3 u, s,
// y in and u, s out; stage 4 u, s, y in and y, comp out (18 transfers).
template <int STAGE, typename C, typename T>
__device__ __forceinline__ void pipe_combine(C* __restrict__ uout, C* __restrict__ accg, C* __restrict__ yg,
                                             C* __restrict__ compg, int gi, C uc, C kv, C sv, C yv, T h2, T hh,
                                             T w_hi, T w_lo) {
  if constexpr (STAGE == 1) {  // sv = comp of the element
    uout[gi] = caxpy(h2, kv, uc);
    accg[gi] = caxpy(w_hi, kv, caxpy(w_lo, kv, cneg(sv)));
  } else if constexpr (STAGE == 2) {
    C ye;
    ye.x = fma((T)-3, sv.x, uc.x);
    ye.y = fma((T)-3, sv.y, uc.y);
    const C k2 = cscale(kv, (T)2);
    uout[gi] = caxpy(h2, kv, ye);
    accg[gi] = caxpy(w_hi, k2, caxpy(w_lo, k2, sv));
  } else if constexpr (STAGE == 3) {
    const C k2 = cscale(kv, (T)2);
    uout[gi] = caxpy(hh, kv, yv);
    accg[gi] = caxpy(w_hi, k2, caxpy(w_lo, k2, sv));
  } else {
    const C p = caxpy(w_hi, kv, caxpy(w_lo, kv, sv));
    C yn, e;
    two_sum(yv, p, yn, e);
    yg[gi] = yn;
    compg[gi] = cneg(e);
  }
}

// State of a pipelined CTA shared by its stage calls: the slots' mbarriers, two batches of
// system records, the stage times and the observable's staging.
template <typename C>
struct PipeShared {
  unsigned long long full[4];
  PipeRec recs[2][BQ_PIPE_RB];  // records of two batches of systems
  double s_t[2];                // physical time of this stage, and of the step midpoint
  float s_t32[2];               // the stage time as an unevaluated FP32 pair (hi, lo)
  C s_of[32];                   // w f_e of the observable entries being evaluated
  C s_ov[6][32];                // y and comp at their G_x, G_y and R points
};

// Once per CTA before its first stage: the slots' mbarriers, and the stage-input region of
// every slot with its guard bands zeroed (neighbour reads at the edges of a system, whose
// coefficients are zero there, land in them, so they must hold finite values; later systems
// leave only earlier systems' finite values behind).
template <typename C>
__device__ __forceinline__ void pipe_init(const PipeArgs& A, PipeShared<C>& sh) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  if (threadIdx.x == 0)
    for (int s = 0; s < A.n_slots; ++s) mbar_init(&sh.full[s], 1);
  for (int s = 0; s < A.n_slots; ++s) {
    float4* z = reinterpret_cast<float4*>(smem_raw + (size_t)s * A.slot_bytes + A.zero_off);
    for (int i = threadIdx.x; i < A.zero_bytes / 16; i += blockDim.x) z[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  fence_proxy_async();  // these writes come before the bulk copies into the same slots
}

// One RK4 stage of every system of this CTA (records blockIdx.x, blockIdx.x + G, ...).  tau:
// tau at the start of the step.  jbase: systems this CTA has put through its slots before
// (system j of this call uses slot (jbase + j) % n_slots and its mbarrier's phase
// ((jbase + j) / n_slots) & 1).  Returns false if a bounded wait gave up (the error word is
// set; the CTA must stop).
template <typename T, int MX, int MY, int MS, int STAGE>
__device__ __forceinline__ bool pipe_stage(const PipeArgs& A, PipeShared<typename C2T<T>::type>& sh, double tau,
                                           int jbase) {
  using C = typename C2T<T>::type;
  constexpr int RS = BQ_PIPE_RS(MS);  // complex entries of a row / column coefficient record
  extern __shared__ __align__(128) unsigned char smem_raw[];
  auto& full = sh.full;
  auto& recs = sh.recs;
  auto& s_t = sh.s_t;

  const int tid = threadIdx.x;
  const int G = gridDim.x;
  const int nj = A.n_sys > (int)blockIdx.x ? (A.n_sys - (int)blockIdx.x + G - 1) / G : 0;
  const int S = A.n_slots;
  const int cs = (int)sizeof(C);
  __syncthreads();  // the previous stage of this CTA is done with the records and times
  if (tid == 0) {
    s_t[0] = pipe_chan_time(1, tau, STAGE, A.dt, A.horizon, A.reverse);
    s_t[1] = pipe_chan_time(2, tau, STAGE, A.dt, A.horizon, A.reverse);
    sh.s_t32[0] = (float)s_t[0];
    sh.s_t32[1] = (float)(s_t[0] - (double)sh.s_t32[0]);
    // the stage input this stage bulk-copies was written by this CTA's threads in its previous
    // stage (generic proxy); order those writes before the copies (async proxy)
    fence_proxy_async_global();
  }
  // FP32: the stage time as an unevaluated FP32 pair, in the threads that load the records
  float t32[2] = {0.f, 0.f};
  if (sizeof(T) == 4 && tid < BQ_PIPE_RB) {
    const double ts = pipe_chan_time(1, tau, STAGE, A.dt, A.horizon, A.reverse);
    t32[0] = (float)ts;
    t32[1] = (float)(ts - (double)t32[0]);
  }
  // a batch of system records; in FP32 each loading thread also evaluates its system's
  // Gaussian envelope at the stage time (as pipe_chan_value does, once per system instead of
  // in every record-building thread ahead of the per-system barrier)
  auto load_batch = [&](int b) {
    if (tid < BQ_PIPE_RB) {
      const int j = b * BQ_PIPE_RB + tid;
      if (j < nj) {
        PipeRec& rr = recs[b & 1][tid];
        rr = A.recs[blockIdx.x + (size_t)j * G];
        if constexpr (sizeof(T) == 4) {
          if (rr.f.gauss) {
            const float d = (t32[0] - rr.f.c_hi) + (t32[1] - rr.f.c_lo);
            const float e = dev_exp<float>(-(d * d) * rr.f.k);
            rr.f.e_re = rr.f.amp_re * e;
            rr.f.e_im = rr.f.amp_im * e;
          }
        }
      }
    }
  };
  load_batch(0);
  __syncthreads();
  auto slot_ptr = [&](int s) { return smem_raw + (size_t)s * A.slot_bytes; };
  // coefficient records of rows and columns, pair-major: pair p (fields 2p, 2p + 1) of row k
  // at rowv[(p BQ_MERGED_MAXM + k) 2], so that lanes with consecutive k or l touch consecutive
  // 16-byte words
  C* rowv = reinterpret_cast<C*>(smem_raw + (size_t)S * A.slot_bytes);  // [RS / 2][BQ_MERGED_MAXM][2]
  C* colv = rowv + (size_t)BQ_MERGED_MAXM * RS;                          // [RS / 2][BQ_MERGED_MAXM][2]

  C* uout = reinterpret_cast<C*>(A.u_out);
  C* yg = reinterpret_cast<C*>(A.y);
  C* accg = reinterpret_cast<C*>(A.acc);
  C* compg = reinterpret_cast<C*>(A.comp);
  const C* uin = reinterpret_cast<const C*>(A.u_in);
  // the array read with per-thread loads besides the stage input: comp at stage 1 (skipped for
  // a freshly loaded state, whose comp is zero), the stage sum otherwise; stages 3 and 4 also
  // read y
  const C* pre = STAGE == 1 ? compg : accg;
  const bool rd = STAGE != 1 || !A.comp_zero;
  constexpr bool RDY = STAGE == 3 || STAGE == 4;

  // thread 0: issue the bulk copies of system j into slot j % S, and bring the arrays this
  // stage reads with per-thread loads into L2, one system ahead of use
  auto issue = [&](int j) {
    const PipeRec& r = recs[(j / BQ_PIPE_RB) & 1][j % BQ_PIPE_RB];
    unsigned char* sl = slot_ptr((jbase + j) % S);
    const unsigned blk = (unsigned)(r.blk_elems * cs);
    fence_proxy_async();
    unsigned long long* bar = &full[(jbase + j) % S];
    mbar_expect_tx(bar, (unsigned)r.param_bytes + blk);
    bulk_g2s(sl, A.params + r.param_off, (unsigned)r.param_bytes, bar);
    bulk_g2s(sl + A.off_u, uin + r.blk_off, blk, bar);
    if (rd) bulk_prefetch_l2(pre + r.blk_off, blk);
    if (RDY) bulk_prefetch_l2(yg + r.blk_off, blk);
  };
  if (tid == 0)
    for (int j = 0; j < S - 1 && j < nj; ++j) issue(j);

  const T hh = (T)A.dt;
  const T h2 = (T)(0.5 * A.dt);
  const double w = A.dt / 6.0;
  const T w_hi = (T)w;
  const T w_lo = (T)(w - (double)w_hi);
  const C zero = cmk<C>(0.0, 0.0);

  // Stage 4: the Tr(rho0 A) contribution of system j (Eqs. 7, 11: w sum_e f_e (G_x[k_e]
  // G_y[l_e] + R[k_e, l_e]) over the entries of rho0's support) from the updated state
  // y - comp, in the state's precision, by warp 1 (lane e: entry e).  No global round trip
  // sits on the warp's path between two barriers: at the end of system j it takes the entries
  // from the parameter block still in slot j (obs_take); after the barrier that makes every
  // thread's writes of system j visible it starts asynchronous copies of the values into
  // shared memory (obs_load, so that no register is held across the next system); they are
  // first read at the end of system j + 1 (obs_give: the products, a shuffle reduction, one
  // store per system).
  const bool obs_on = STAGE == 4 && A.obs != nullptr && (tid >> 5) == 1;
  auto& s_of = sh.s_of;  // w f_e of the entries being evaluated
  auto& s_ov = sh.s_ov;  // y and comp at their G_x, G_y and R points
  int oa = -1, ob = -1, oc = -1, on = 0;
  auto obs_take = [&](int j) {
    const PipeRec& rj = recs[(j / BQ_PIPE_RB) & 1][j % BQ_PIPE_RB];
    const unsigned char* sj = slot_ptr((jbase + j) % S);
    const PipeHdr& hj = *reinterpret_cast<const PipeHdr*>(sj);
    const int lane = tid & 31;
    on = hj.n_obs;
    oa = ob = oc = -1;
    if (lane < on) {
      const PipeObs<C>& en = reinterpret_cast<const PipeObs<C>*>(sj + hj.obs_off)[lane];
      if (rj.gy_off >= 0) {
        oa = rj.blk_off + en.kx;
        ob = rj.blk_off + rj.gy_off + en.ly;
      }
      if (rj.r_off >= 0) oc = rj.blk_off + rj.r_off + en.kx * rj.M + en.ly;
      C w;
      if constexpr (sizeof(T) == 8) w = cmk<C>(rj.d.w_re, rj.d.w_im);
      else w = make_float2(rj.w32_re, rj.w32_im);
      s_of[lane] = cmul(w, en.f);
    }
  };
  auto obs_load = [&]() {
    const int lane = tid & 31;
    if (oa >= 0) {
      cp_async_c(&s_ov[0][lane], yg + oa);
      cp_async_c(&s_ov[1][lane], compg + oa);
      cp_async_c(&s_ov[2][lane], yg + ob);
      cp_async_c(&s_ov[3][lane], compg + ob);
    }
    if (oc >= 0) {
      cp_async_c(&s_ov[4][lane], yg + oc);
      cp_async_c(&s_ov[5][lane], compg + oc);
    }
    cp_async_commit();
  };
  auto obs_give = [&](int j) {
    const int lane = tid & 31;
    cp_async_wait_all();
    C v = zero;
    if (oa >= 0) v = cmul(cadd(s_ov[0][lane], cneg(s_ov[1][lane])), cadd(s_ov[2][lane], cneg(s_ov[3][lane])));
    if (oc >= 0) v = cadd(v, cadd(s_ov[4][lane], cneg(s_ov[5][lane])));
    C c = lane < on ? cmul(s_of[lane], v) : zero;
    if (on > 1) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        c.x += __shfl_down_sync(0xffffffffu, c.x, o);
        c.y += __shfl_down_sync(0xffffffffu, c.y, o);
      }
    }
    if (lane == 0) A.obs[recs[(j / BQ_PIPE_RB) & 1][j % BQ_PIPE_RB].sys] = make_double2((double)c.x, (double)c.y);
  };
  auto obs_end = [&](int j) {
    if (!obs_on) return;
    if (j > 0) obs_give(j - 1);
    obs_take(j);
  };

  for (int j = 0; j < nj; ++j) {
    const int jn = j + S - 1;
    if (jn < nj && jn % BQ_PIPE_RB == 0) {
      load_batch(jn / BQ_PIPE_RB);
      __syncthreads();
    }
    const PipeRec r = recs[(j / BQ_PIPE_RB) & 1][j % BQ_PIPE_RB];
    const int M = r.M;
    const int gb = r.blk_off;
    const bool merged = r.merged != 0;
    // Merged path: this thread's column strip (column l, rows k0..k1-1 of R) and its G item
    // (index gq of [G_x | G_y], handed out from the last thread down, where the strips are
    // shortest or absent).  The streamed values of the strip's first two rows and of the G
    // item are loaded before the wait for the stage input.
    int l = 0, k0 = 0, k1 = 0, gq = -1, gg = 0;
    C s0 = zero, s1 = zero, y0 = zero, y1 = zero, sG = zero, yG = zero;
    if (merged) {
      const int bk = (int)(((float)tid + 0.5f) * r.inv_m);
      l = tid - bk * M;
      if (r.r_off >= 0 && bk < r.nb) {
        k0 = bk * r.rb;
        k1 = min(M, k0 + r.rb);
      }
      const int gi_ = BQ_PIPE_THREADS - 1 - tid;
      if (r.gy_off >= 0 && gi_ < 2 * M) {
        gq = gi_;
        gg = gb + (gq < M ? gq : r.gy_off + gq - M);
        if (rd) sG = pre[gg];
        if (RDY) yG = yg[gg];
      }
      const int g0 = gb + r.r_off + k0 * M + l;
      if (k0 < k1) {
        if (rd) s0 = pre[g0];
        if (RDY) y0 = yg[g0];
      }
      if (k0 + 1 < k1) {
        if (rd) s1 = pre[g0 + M];
        if (RDY) y1 = yg[g0 + M];
      }
    }
    const bool rowb = merged && tid < M;
    const bool colb = merged && tid >= BQ_MERGED_MAXM && tid - BQ_MERGED_MAXM < M;
    // wait for system j (bounded): one thread polls the mbarrier, the others wait at the
    // barrier without issuing; the completed phase also makes the bulk-copied data visible
    {
      bool ok = true;
      if (tid == 0) {
        ok = false;
        for (int it = 0; it < BQ_WAIT_SUSPENDS; ++it)
          if (mbar_try_wait_for(&full[(jbase + j) % S], (unsigned)(((jbase + j) / S) & 1), BQ_WAIT_HINT_NS)) {
            ok = true;
            break;
          }
      }
      if (__syncthreads_or(!ok)) {
        if (tid == 0) atomicOr(A.error, 1u);
        // give the copies in flight a bounded chance to land before the CTA leaves
        for (int s = 0; s < S; ++s)
          for (int it = 0; it < BQ_WAIT_LIMIT; ++it)
            if (mbar_try_wait(&full[s], (unsigned)(((jbase + j) / S) & 1))) break;
        return false;
      }
    }
    // every thread is past system j - 1: its slot ((j + S - 1) % S) and the coefficient
    // records are free, so the next copy can start now
    if (tid == 0 && jn < nj) issue(jn);
    if (obs_on && j > 0) obs_load();
    unsigned char* sl = slot_ptr((jbase + j) % S);
    const PipeHdr& h = *reinterpret_cast<const PipeHdr*>(sl);
    const int nX = h.nX, nY = h.nY, nS = h.nS, has_sep = h.has_sep;
    const int sdiag = h.sdiag;  // bit q: sandwich term q acts only where k = l
    const PipeCoef<C>* tc = reinterpret_cast<const PipeCoef<C>*>(sl + sizeof(PipeHdr));
    const PipeChan* pc = reinterpret_cast<const PipeChan*>(tc + h.n_terms);
    const C* dx = reinterpret_cast<const C*>(pc + h.n_ch);
    const C* dy = dx + M;
    const T* wX = reinterpret_cast<const T*>(dy + M);
    const T* wY = wX + nX * M;
    const T* wSx = wY + nY * M;
    const T* wSy = wSx + nS * M;
    const C* u = reinterpret_cast<const C*>(sl + A.off_u);
    const C* ur = u + r.r_off;
    const C* ugx = u;
    const C* ugy = u + r.gy_off;
    C Cc;
    if constexpr (sizeof(T) == 8) Cc = cmk<C>(r.d.c_re, r.d.c_im);
    else Cc = make_float2(r.c32_re, r.c32_im);
    // drive envelopes of the problem's time-dependent terms at this stage's time, from the
    // block (threads that build coefficient records; every thread on the general path)
    C e0 = cmk<C>(1.0, 0.0), e1 = cmk<C>(1.0, 0.0);
    if (!merged || rowb || colb) {
      bool pre_e = false;
      if constexpr (sizeof(T) == 4) {
        if (r.f.gauss) {  // evaluated with the batch of records
          e0 = make_float2(r.f.e_re, r.f.e_im);
          pre_e = true;
        }
      }
      if (!pre_e) {
        if (h.n_ch > 0) e0 = pipe_chan_value<T>(pc[0], A.chpar, s_t[0], s_t[1], sh.s_t32);
        if (h.n_ch > 1) e1 = pipe_chan_value<T>(pc[1], A.chpar, s_t[0], s_t[1], sh.s_t32);
      }
    }
    // stage coefficient of term q: static part times the envelope (or its conjugate)
    auto coef = [&](int q) {
      const C c = tc[q].c;
      const int ch = tc[q].ch;
      if (ch < 0) return c;
      C e = ch == 0 ? e0 : e1;
      if (tc[q].conj) e.y = -e.y;
      return cmul(c, e);
    };
    const int nr = h.has_r ? M * M : 0;
    const int ntot = h.ntot;

    if (merged) {
      // ---- merged stencil: per-row / per-column coefficient records, one strip per thread ----
      // row record k: A0 (diagonal + shift-0 X terms), Am (shift -1), Ap (shift +1), then per
      // sandwich term q with shifts (sx, sy): SX_q = c_q Wx_q[k] and SG_q = SX_q G_x[k + sx];
      // column record l: B0, Bm, Bp of the Y terms, then SY_q = Wy_q[l] (real part) and
      // GY_q = Wy_q[l] G_y[l + sy].  A point (k, l) of R gets
      //   (A0 + B0) u + Am u(k-1,l) + Ap u(k+1,l) + Bm u(k,l-1) + Bp u(k,l+1)
      //   + sum_q SX_q SY_q u(k+sx,l+sy) + SG_q GY_q,
      // without bounds tests: every coefficient whose source leaves the grid is zero and the
      // source read itself stays inside the slot's guard bands.
      if (rowb) {
        const int i = tid;
        C a0 = dx[i], am = zero, ap = zero;
#pragma unroll
        for (int q = 0; q < MX; ++q)
          if (q < nX) {
            const C v = cscale(coef(q), wX[q * M + i]);
            if (h.sX[q] == 0) a0 = cadd(a0, v); else if (h.sX[q] < 0) am = cadd(am, v); else ap = cadd(ap, v);
          }
        C f[RS];
        f[0] = a0; f[1] = am; f[2] = ap;
#pragma unroll
        for (int q = 0; q < MS; ++q) {
          f[3 + 2 * q] = zero;
          f[4 + 2 * q] = zero;
          if (q < nS) {
            const C sx = cscale(coef(nX + nY + q), wSx[q * M + i]);
            const int xs = i + h.sSx[q];
            const C gx = (has_sep && xs >= 0 && xs < M) ? ugx[xs] : zero;
            f[3 + 2 * q] = sx;
            f[4 + 2 * q] = cmul(sx, gx);
          }
        }
        if (RS > 3 + 2 * MS) f[RS - 1] = zero;
#pragma unroll
        for (int p = 0; p < RS / 2; ++p) st_pair(rowv + (p * BQ_MERGED_MAXM + i) * 2, f[2 * p], f[2 * p + 1]);
      } else if (colb) {
        const int i = tid - BQ_MERGED_MAXM;
        C b0 = dy[i], bm = zero, bp = zero;
#pragma unroll
        for (int q = 0; q < MY; ++q)
          if (q < nY) {
            const C v = cscale(coef(nX + q), wY[q * M + i]);
            if (h.sY[q] == 0) b0 = cadd(b0, v); else if (h.sY[q] < 0) bm = cadd(bm, v); else bp = cadd(bp, v);
          }
        C f[RS];
        f[0] = b0; f[1] = bm; f[2] = bp;
#pragma unroll
        for (int q = 0; q < MS; ++q) {
          f[3 + 2 * q] = zero;
          f[4 + 2 * q] = zero;
          if (q < nS) {
            const T wy = wSy[q * M + i];
            const int ys = i + h.sSy[q];
            f[3 + 2 * q].x = wy;
            if (has_sep && ys >= 0 && ys < M) f[4 + 2 * q] = cscale(ugy[ys], wy);
          }
        }
        if (RS > 3 + 2 * MS) f[RS - 1] = zero;
#pragma unroll
        for (int p = 0; p < RS / 2; ++p) st_pair(colv + (p * BQ_MERGED_MAXM + i) * 2, f[2 * p], f[2 * p + 1]);
      }
      __syncthreads();
      // the strip loop, compiled for the system's number of sandwich terms NS (the per-point
      // term loop then has no runtime bound)
      auto strip = [&](auto ns_c) {
        constexpr int NS = decltype(ns_c)::value;
        // field f of column l's record: pair f / 2, half f % 2
        auto cfld = [&](int f) { return colv[((f >> 1) * BQ_MERGED_MAXM + l) * 2 + (f & 1)]; };
        const C b0 = cfld(0), bm = cfld(1), bp = cfld(2);
        T syq[NS > 0 ? NS : 1];
        C gyq[NS > 0 ? NS : 1];
        int soff[NS > 0 ? NS : 1];
        bool sdq[NS > 0 ? NS : 1];
#pragma unroll
        for (int q = 0; q < NS; ++q) {
          syq[q] = cfld(3 + 2 * q).x;
          gyq[q] = cfld(4 + 2 * q);
          soff[q] = h.sSx[q] * M + h.sSy[q];
          sdq[q] = (sdiag >> q) & 1;
        }
        const C* up = ur + k0 * M + l;  // the point (kk, l)
        const C* rv = rowv + k0 * 2;     // pair 0 of row kk's record
        int go = gb + r.r_off + k0 * M + l;
        C um = up[-M];  // (k0 - 1, l): the row above, or a guard / G value with Am = 0
        C uc = up[0];
        // the stencil of one point from its row record (pair p at rrec + 2 p BQ_MERGED_MAXM)
        // and the column values in registers.  The row-neighbour, column-neighbour and
        // sandwich parts are summed in independent chains and the row and column parts added
        // to each other before the diagonal part: a point and its mirror (l, k) then round
        // alike, so R keeps the conjugate symmetry of a Hermitian operator's expansion.
        constexpr int PS = 2 * BQ_MERGED_MAXM;
        auto point = [&](const C* rrec, const C* pu, C cm, C cc, C cd, bool on_diag) {
          C a0, am, ap, sxn;
          ld_pair(rrec, a0, am);
          ld_pair(rrec + PS, ap, sxn);
          const C kd = cmul(cadd(a0, b0), cc);
          C kr = cmul(am, cm);
          C kc = cmul(bm, pu[-1]);
          kr = cfma(ap, cd, kr);
          kc = cfma(bp, pu[1], kc);
          C ks = zero;
#pragma unroll
          for (int q = 0; q < NS; ++q) {
            const C sx = sxn;
            C sg;
            ld_pair(rrec + (2 + q) * PS, sg, sxn);
            if (!sdq[q] || on_diag) {  // secular projector: k = l only
              ks = cfma(cscale(sx, syq[q]), pu[soff[q]], ks);
              ks = cfma(sg, gyq[q], ks);
            }
          }
          return cadd(cadd(kd, cadd(kr, kc)), ks);
        };
        // two rows per iteration (independent chains); streamed values in a register ring
        // two rows ahead of use
        for (int kk = k0; kk < k1; kk += 2) {
          const bool two = kk + 1 < k1;
          const C sA = s0, yA = y0, sB = s1, yB = y1;
          if (kk + 2 < k1) {
            if (rd) s0 = pre[go + 2 * M];
            if (RDY) y0 = yg[go + 2 * M];
          }
          if (kk + 3 < k1) {
            if (rd) s1 = pre[go + 3 * M];
            if (RDY) y1 = yg[go + 3 * M];
          }
          const C ud = up[M];                     // row kk + 1 (a guard row past M - 1)
          const C udB = two ? up[2 * M] : zero;   // row kk + 2 (at most row M: the guard band)
          const C kvA = point(rv, up, um, uc, ud, kk == l);
          pipe_combine<STAGE>(uout, accg, yg, compg, go, uc, kvA, sA, yA, h2, hh, w_hi, w_lo);
          if (two) {
            const C kvB = point(rv + 2, up + M, uc, ud, udB, kk + 1 == l);
            pipe_combine<STAGE>(uout, accg, yg, compg, go + M, ud, kvB, sB, yB, h2, hh, w_hi, w_lo);
          }
          um = ud;
          uc = udB;
          up += 2 * M;
          rv += 4;
          go += 2 * M;
        }
      };
      // (a system without sandwich terms takes the one-term loop: the builders zero-fill the
      // unused record fields, so the extra term adds exact zeros; fewer loop copies keep the
      // kernel's code small)
      if (k0 < k1) {
        if (nS <= 1) strip(std::integral_constant<int, 1>{});
        else if (nS == 2 || MS == 2) strip(std::integral_constant<int, (MS >= 2 ? 2 : 1)>{});
        else strip(std::integral_constant<int, MS>{});
      }
      if (gq >= 0) {
        const bool isx = gq < M;
        const int g = isx ? gq : gq - M;
        const C* gs = isx ? ugx : ugy;
        const C* vv = (isx ? rowv : colv) + g * 2;  // fields 0, 1 (pair 0) and 2 (pair 1)
        const C uc = gs[g];
        // neighbours outside the grid have zero coefficients; their reads stay in the slot
        const C lo = gs[g - 1], hi = gs[g + 1];
        C d = vv[0];
        d = isx ? cadd(d, Cc) : cadd(d, cneg(Cc));
        C kv = cmul(d, uc);
        kv = cfma(vv[1], lo, kv);
        kv = cfma(vv[2 * BQ_MERGED_MAXM], hi, kv);
        pipe_combine<STAGE>(uout, accg, yg, compg, gg, uc, kv, sG, yG, h2, hh, w_hi, w_lo);
      }
      obs_end(j);
      // no barrier here: the wait at the top of the next system orders the reuse of the
      // slot and of the coefficient records
      continue;
    }

    // ---- general term program (any shifts) ----------------------------------------------
    C cX[MX], cY[MY], cS[MS];
    int shX[MX], shY[MY], shSx[MS], shSy[MS];
#pragma unroll
    for (int q = 0; q < MX; ++q) { cX[q] = q < nX ? coef(q) : zero; shX[q] = h.sX[q]; }
#pragma unroll
    for (int q = 0; q < MY; ++q) { cY[q] = q < nY ? coef(nX + q) : zero; shY[q] = h.sY[q]; }
#pragma unroll
    for (int q = 0; q < MS; ++q) {
      cS[q] = q < nS ? coef(nX + nY + q) : zero;
      shSx[q] = h.sSx[q];
      shSy[q] = h.sSy[q];
    }
    const float invM = r.inv_m;
    for (int e = tid; e < ntot; e += blockDim.x) {
      int pos;
      C uc, kv;
      if (e < nr) {
        const int kx = (int)(((float)e + 0.5f) * invM);
        const int ly = e - kx * M;
        pos = r.r_off + e;
        uc = ur[e];
        kv = cmul(cadd(dx[kx], dy[ly]), uc);
#pragma unroll
        for (int q = 0; q < MX; ++q)
          if (q < nX) kv = cfma(cX[q], cscale(ur[min(max(kx + shX[q], 0), M - 1) * M + ly], wX[q * M + kx]), kv);
#pragma unroll
        for (int q = 0; q < MY; ++q)
          if (q < nY) kv = cfma(cY[q], cscale(ur[kx * M + min(max(ly + shY[q], 0), M - 1)], wY[q * M + ly]), kv);
#pragma unroll
        for (int q = 0; q < MS; ++q)
          if (q < nS && (!((sdiag >> q) & 1) || kx == ly)) {  // secular projector: k = l only
            const int rr = min(max(kx + shSx[q], 0), M - 1);
            const int cc = min(max(ly + shSy[q], 0), M - 1);
            C v = ur[rr * M + cc];
            if (has_sep) v = cadd(v, cmul(ugx[rr], ugy[cc]));
            kv = cfma(cS[q], cscale(v, wSx[q * M + kx] * wSy[q * M + ly]), kv);
          }
      } else {
        const bool isx = e < nr + M;
        const int g = isx ? e - nr : e - nr - M;
        const C* gs = isx ? ugx : ugy;
        pos = isx ? g : r.gy_off + g;
        uc = gs[g];
        kv = cmul(isx ? cadd(dx[g], Cc) : cadd(dy[g], cneg(Cc)), uc);
        if (isx) {
#pragma unroll
          for (int q = 0; q < MX; ++q)
            if (q < nX) kv = cfma(cX[q], cscale(gs[min(max(g + shX[q], 0), M - 1)], wX[q * M + g]), kv);
        } else {
#pragma unroll
          for (int q = 0; q < MY; ++q)
            if (q < nY) kv = cfma(cY[q], cscale(gs[min(max(g + shY[q], 0), M - 1)], wY[q * M + g]), kv);
        }
      }
      const int gi = gb + pos;
      const C sv = rd ? pre[gi] : zero;
      const C yv = RDY ? yg[gi] : zero;
      pipe_combine<STAGE>(uout, accg, yg, compg, gi, uc, kv, sv, yv, h2, hh, w_hi, w_lo);
    }
    obs_end(j);
  }
  __syncthreads();  // every system of this CTA is written (and its slots are free)
  if (obs_on && nj > 0) {
    obs_load();
    obs_give(nj - 1);
  }
  return true;
}

// The last CTA to finish advances the state's step counter by n.
__device__ __forceinline__ void pipe_ticket(const PipeArgs& A, long long n) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned int t = atomicAdd(A.ticket, 1u);
    if (t == gridDim.x - 1) {
      *A.ticket = 0u;
      *A.counter = *(volatile long long*)A.counter + n;
      __threadfence();
    }
  }
}

// One stage launch.
template <typename T, int MX, int MY, int MS, int STAGE>
__global__ void __launch_bounds__(BQ_PIPE_THREADS) k_stage_pipe(const PipeArgs A) {
  __shared__ PipeShared<typename C2T<T>::type> sh;
  pipe_init(A, sh);
  const double tau = A.tau_base[0] + (double)(*(volatile long long*)A.counter) * A.dt;
  if (!pipe_stage<T, MX, MY, MS, STAGE>(A, sh, tau, 0)) return;
  if (STAGE == 4) pipe_ticket(A, 1);
}

// n_steps RK4 steps in one launch.  A system's stage depends only on the same system's
// previous stage, and every CTA owns the same systems in every stage, so the CTAs never wait
// for one another: each runs its systems' stages in order (the stage inputs alternate
// between ua and ub as in the per-stage launches) while the other CTAs are at other stages.
// bq_step launches it one step at a time (the CTAs then drift apart by at most a step).
template <typename T, int MX, int MY, int MS>
__global__ void __launch_bounds__(BQ_PIPE_THREADS) k_steps_pipe(const PipeArgs A, void* ua, void* ub, int n_steps) {
  __shared__ PipeShared<typename C2T<T>::type> sh;
  pipe_init(A, sh);
  const int G = gridDim.x;
  const int nj = A.n_sys > (int)blockIdx.x ? (A.n_sys - (int)blockIdx.x + G - 1) / G : 0;
  const double tau0 = A.tau_base[0] + (double)(*(volatile long long*)A.counter) * A.dt;
  int jbase = 0;
  for (int i = 0; i < n_steps; ++i) {
    const double tau = tau0 + (double)i * A.dt;
    PipeArgs a = A;
    a.comp_zero = i == 0 ? A.comp_zero : 0;
    a.obs = nullptr;
    a.u_in = A.y; a.u_out = ua;
    if (!pipe_stage<T, MX, MY, MS, 1>(a, sh, tau, jbase)) return;
    jbase += nj;
    a.u_in = ua; a.u_out = ub;
    if (!pipe_stage<T, MX, MY, MS, 2>(a, sh, tau, jbase)) return;
    jbase += nj;
    a.u_in = ub; a.u_out = ua;
    if (!pipe_stage<T, MX, MY, MS, 3>(a, sh, tau, jbase)) return;
    jbase += nj;
    a.u_in = ua; a.u_out = nullptr;
    a.obs = i == n_steps - 1 ? A.obs : nullptr;  // the observable of the last step
    if (!pipe_stage<T, MX, MY, MS, 4>(a, sh, tau, jbase)) return;
    jbase += nj;
  }
  pipe_ticket(A, n_steps);
}


// ---------------------------------------------------------------------------------------
// Batched persistent solve (single mode): one launch integrates every system for n_steps.
// Each CTA takes systems from an atomic queue (largest first), keeps the two RK4 stage
// buffers [R | G_x | G_y] in shared memory and the state y, the stage sum and the
// rounding compensation of the points it owns in registers, and runs all steps with one
// barrier per stage.  Drive coefficients of the next stage are evaluated by a few threads
// while the others compute.  There is no inter-CTA waiting of any kind.
// ---------------------------------------------------------------------------------------
template <typename T, int BLK, int PPT, int MX, int MY, int MS, bool DIAG>
__global__ void __launch_bounds__(BLK, 2) k_solve_m1(const SolveArgs A) {
  using C = typename C2T<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ M1Sys s;
  __shared__ C coef[2][3 * BQ_M1_MAXT];
  __shared__ int s_next;
  const int tid = threadIdx.x;
  C* y_g = reinterpret_cast<C*>(A.y);
  C* comp_g = reinterpret_cast<C*>(A.comp);

  for (;;) {
    if (tid == 0) s_next = (int)atomicAdd(A.queue, 1u);
    __syncthreads();
    const int qi = s_next;
    if (qi >= A.n_sys) return;
    {
      const int* src = reinterpret_cast<const int*>(A.m1 + A.order[qi]);
      int* dst = reinterpret_cast<int*>(&s);
      for (int i = tid; i < (int)(sizeof(M1Sys) / sizeof(int)); i += BLK) dst[i] = src[i];
    }
    __syncthreads();
    const int M = s.M, nX = s.nX, nY = s.nY, nS = s.nS;
    const int sdiag = s.sdiag;  // bit q: sandwich term q acts only where k = l
    const int has_r = s.has_r, has_sep = s.has_sep;
    const int nr = has_r ? M * M : 0;
    const int ntot = nr + (has_sep ? 2 * M : 0);
    // shared: B0[ntot] | B1[ntot] | dx[M] | dy[M] | weights (real)
    C* B0 = reinterpret_cast<C*>(smem_raw);
    C* B1 = B0 + ntot;
    C* dx = B1 + ntot;
    C* dy = dx + M;
    T* wX = reinterpret_cast<T*>(dy + M);
    T* wY = wX + nX * M;
    T* wSx = wY + nY * M;
    T* wSy = wSx + nS * M;
    const int nt = nX + nY + nS;
    auto eval_coef = [&](int buf, int64_t step, int stage) {
      if (tid < nt) {
        const int t = tid < nX ? s.tX[tid] : (tid < nX + nY ? s.tY[tid - nX] : s.tS[tid - nX - nY]);
        const TermDesc& td = A.terms[s.term_off + t];
        double2 c = make_double2(td.c_re, td.c_im);
        if (td.ch >= 0) {
          const ChanDesc cd = A.chans[td.ch];
          const double ts = A.tau0 + (double)step * A.dt;
          const double tau = (cd.kind == 2) ? ts + 0.5 * A.dt : ts + stage_c(stage) * A.dt;
          double2 e = chan_value_t<T>(cd, A.chpar, A.reverse ? A.horizon - tau : tau);
          if (td.conj) e.y = -e.y;
          c = make_double2(c.x * e.x - c.y * e.y, c.x * e.y + c.y * e.x);
        }
        coef[buf][tid] = cmk<C>(c.x, c.y);
      }
    };
    // global index of element e of [R | G_x | G_y]
    auto gidx = [&](int e) -> int64_t {
      return e < nr ? s.off_r + e : (e < nr + M ? s.off_gx + (e - nr) : s.off_gy + (e - nr - M));
    };
    C yv[PPT], av[PPT], cv[PPT];
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
      const int e = tid + j * BLK;
      if (e < ntot) {
        const int64_t g = gidx(e);
        yv[j] = y_g[g];
        cv[j] = comp_g[g];
        B0[e] = yv[j];
      }
    }
    {
      const C* Dg = reinterpret_cast<const C*>(A.diag) + s.diag_off;
      const T* W = reinterpret_cast<const T*>(A.wtab);
      for (int i = tid; i < M; i += BLK) {
        dx[i] = Dg[i];
        dy[i] = Dg[M + i];
#pragma unroll
        for (int j = 0; j < MX; ++j) if (j < nX) wX[j * M + i] = s.wX[j] >= 0 ? W[s.wX[j] + i] : (T)1;
#pragma unroll
        for (int j = 0; j < MY; ++j) if (j < nY) wY[j * M + i] = s.wY[j] >= 0 ? W[s.wY[j] + i] : (T)1;
#pragma unroll
        for (int j = 0; j < MS; ++j)
          if (j < nS) {
            wSx[j * M + i] = s.wSx[j] >= 0 ? W[s.wSx[j] + i] : (T)1;
            wSy[j * M + i] = s.wSy[j] >= 0 ? W[s.wSy[j] + i] : (T)1;
          }
      }
    }
    eval_coef(0, 0, 1);
    int shX[MX], shY[MY], shSx[MS], shSy[MS];
#pragma unroll
    for (int j = 0; j < MX; ++j) shX[j] = s.sX[j];
#pragma unroll
    for (int j = 0; j < MY; ++j) shY[j] = s.sY[j];
#pragma unroll
    for (int j = 0; j < MS; ++j) { shSx[j] = s.sSx[j]; shSy[j] = s.sSy[j]; }
    const C Cc = cmk<C>(s.c_re, s.c_im);
    const T dt = (T)A.dt;
    const float invM = 1.0f / (float)M;
    __syncthreads();

    int buf = 0;
    for (int64_t step = 0; step < A.n_steps; ++step) {
#pragma unroll 1
      for (int stage = 1; stage <= 4; ++stage) {
        const C* uin = (stage & 1) ? B0 : B1;  // stages 1, 3 read B0; 2, 4 read B1
        C* uout = (stage & 1) ? B1 : B0;
        C cX[MX], cY[MY], cS[MS];
#pragma unroll
        for (int j = 0; j < MX; ++j) cX[j] = coef[buf][min(j, 3 * BQ_M1_MAXT - 1)];
#pragma unroll
        for (int j = 0; j < MY; ++j) cY[j] = coef[buf][min(nX + j, 3 * BQ_M1_MAXT - 1)];
#pragma unroll
        for (int j = 0; j < MS; ++j) cS[j] = coef[buf][min(nX + nY + j, 3 * BQ_M1_MAXT - 1)];
        const C* gxi = uin + nr;
        const C* gyi = gxi + M;
#pragma unroll
        for (int j = 0; j < PPT; ++j) {
          const int e = tid + j * BLK;
          if (e >= ntot) continue;
          const C uc = uin[e];
          C kv;
          if (e < nr) {
            const int kx = (int)(((float)e + 0.5f) * invM);
            const int ly = e - kx * M;
            kv = cmul(cadd(dx[kx], dy[ly]), uc);
#pragma unroll
            for (int q = 0; q < MX; ++q)
              if (q < nX) kv = cfma(cX[q], cscale(uin[min(max(kx + shX[q], 0), M - 1) * M + ly], wX[q * M + kx]), kv);
#pragma unroll
            for (int q = 0; q < MY; ++q)
              if (q < nY) kv = cfma(cY[q], cscale(uin[kx * M + min(max(ly + shY[q], 0), M - 1)], wY[q * M + ly]), kv);
#pragma unroll
            for (int q = 0; q < MS; ++q)
              if (q < nS && (!DIAG || !((sdiag >> q) & 1) || kx == ly)) {  // secular projector: k = l only
                const int r = min(max(kx + shSx[q], 0), M - 1);
                const int c = min(max(ly + shSy[q], 0), M - 1);
                C v = uin[r * M + c];
                if (has_sep) v = cadd(v, cmul(gxi[r], gyi[c]));
                kv = cfma(cS[q], cscale(v, wSx[q * M + kx] * wSy[q * M + ly]), kv);
              }
          } else {
            const bool isx = e < nr + M;
            const int g = isx ? e - nr : e - nr - M;
            const C* gs = isx ? gxi : gyi;
            kv = cmul(isx ? cadd(dx[g], Cc) : cadd(dy[g], cmk<C>(-s.c_re, -s.c_im)), uc);
            if (isx) {
#pragma unroll
              for (int q = 0; q < MX; ++q)
                if (q < nX) kv = cfma(cX[q], cscale(gs[min(max(g + shX[q], 0), M - 1)], wX[q * M + g]), kv);
            } else {
#pragma unroll
              for (int q = 0; q < MY; ++q)
                if (q < nY) kv = cfma(cY[q], cscale(gs[min(max(g + shY[q], 0), M - 1)], wY[q * M + g]), kv);
            }
          }
          // RK4 combine (stage sum + compensated state update, as in the stage kernels)
          if (stage == 1) {
            uout[e] = caxpy(dt * (T)0.5, kv, yv[j]);
            av[j] = kv;
          } else if (stage == 4) {
            const C sm = cadd(av[j], kv);
            C d, t;
            d.x = dt * (T)(1.0 / 6.0) * sm.x - cv[j].x;
            d.y = dt * (T)(1.0 / 6.0) * sm.y - cv[j].y;
            t.x = yv[j].x + d.x;
            t.y = yv[j].y + d.y;
            cv[j].x = (t.x - yv[j].x) - d.x;
            cv[j].y = (t.y - yv[j].y) - d.y;
            yv[j] = t;
            uout[e] = t;
          } else {
            uout[e] = caxpy(stage == 2 ? dt * (T)0.5 : dt, kv, yv[j]);
            av[j] = caxpy((T)2, kv, av[j]);
          }
        }
        // coefficients of the next stage (stage 4 -> stage 1 of the next step)
        const int nstage = stage == 4 ? 1 : stage + 1;
        eval_coef(buf ^ 1, stage == 4 ? step + 1 : step, nstage);
        buf ^= 1;
        __syncthreads();
      }
    }
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
      const int e = tid + j * BLK;
      if (e < ntot) {
        const int64_t g = gidx(e);
        y_g[g] = yv[j];
        comp_g[g] = cv[j];
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------
// Adjoint (backward-in-time) RK4 stage: the exact discrete adjoint of the stage kernels.
//
// For stage i of a step with cotangent lam of the state after the step:
//   q_i = J_i^T b_i, lacc += q_i (lacc = lam + q_4 at stage 4),
//   b_{i-1} = dt beta_{i-1} lam + c_i dt q_i  (beta = 1/6, 1/3, 1/3; c = 1/2, 1/2, 1 for i = 2, 3, 4),
//   dl/dtheta += Re <b_i, df/dtheta(u_i)> (bilinear pairing, the system is complex linear).
// J^T of a stencil term  out[p] += c W(p) u[p + delta]  is the gather
//   q[p] += c W(p - delta) b[p - delta]  (source point inside the grid),
// and <b, T_t u> = <T_t^T b, u>, so the parameter sums need u only at the point itself.
// The transposed separable source uses the reductions of k_adj_src.
// ---------------------------------------------------------------------------------------
#define BQ_MAX_GT 16  // gradient terms whose sums a thread keeps in registers

__device__ __forceinline__ int pwc_segment(const ChanDesc& cd, const double* par, double t) {
  const double* p = par + cd.par_off;
  const int n_seg = (cd.n_par - 2) / 2;
  const double x = floor((t - p[0]) / p[1]);
  if (!(x >= 0.0) || x >= (double)n_seg) return -1;
  return (int)x;
}

// (a call: inlined, it costs the callers registers on the path of the usual 16 terms or fewer)
__device__ __noinline__ void add_shared(double* to, double x, double y) {
  atomicAdd(to, x);
  atomicAdd(to + 1, y);
}

// One work item of an adjoint stage (k_adj_stage: one per CTA; the cooperative backward
// segment kernel: the CTA's items of every stage); fresh as in stage_body.  gacc / dcacc: the
// calling thread's partial gradient sums, owned by the caller.  With accumulate, they carry
// over to the CTA's next call (same item) and are reduced into the gradient slots only when
// a term's factor changes before that call (a time-dependent envelope other than a piecewise
// constant one, or a new piecewise-constant segment) or when last; otherwise every call
// reduces them.
template <typename T, int NM>
__device__ __forceinline__ void adj_stage_body(const AdjArgs& A, int item, bool fresh, double2 (&gacc)[BQ_MAX_GT],
                                               double2& dcacc, bool accumulate, bool last) {
  using C = typename C2T<T>::type;
  constexpr int ND = 2 * NM;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* bw = reinterpret_cast<C*>(smem_raw);
  __shared__ SysDesc sd;
  __shared__ WorkItem wi;
  __shared__ TermDesc st[BQ_MAX_TERMS];
  __shared__ C sc[BQ_MAX_TERMS];
  __shared__ int gidx[BQ_MAX_TERMS];
  __shared__ int s_ngt, s_nS;
  __shared__ int sidx[BQ_MAX_TERMS];       // ordinal of an S term
  __shared__ double red[BQ_BLOCK / 32][2 * BQ_MAX_GT + 2];  // per-warp sums of the gradient terms
  // sums of the gradient terms beyond BQ_MAX_GT (rare: 17 and more); zero except between a call that
  // keeps its sums and the CTA's next
  __shared__ double more[2 * (BQ_MAX_TERMS - BQ_MAX_GT)];

  const int tid = threadIdx.x;
  const int stage = A.stage;
  __syncthreads();  // the CTA's previous item is done with the shared copies
  if (fresh)
    for (int i = tid; i < 2 * (BQ_MAX_TERMS - BQ_MAX_GT); i += blockDim.x) more[i] = 0.0;
  if (tid == 0 && fresh) {
    wi = A.work[item];
    sd = A.sys[wi.sys];
  }
  __syncthreads();
  const int nt = sd.n_terms;
  for (int t = tid; t < nt; t += blockDim.x) {
    if (fresh) st[t] = A.terms[sd.term_off + t];
    const double2 c = term_coef(st[t], A.chans, A.chpar, A.tau_step, A.dt, stage, A.horizon, A.reverse);
    sc[t] = cmk<C>(c.x, c.y);
  }
  if (tid == 0 && fresh) {
    int g = 0, s = 0;
    for (int t = 0; t < nt; ++t) {
      const TermDesc& td = A.terms[sd.term_off + t];
      gidx[t] = td.gslot_param >= 0 || td.gslot_pwc >= 0 ? g++ : -1;
      sidx[t] = td.side == SIDE_S ? s++ : -1;
    }
    s_ngt = g;
    s_nS = s;
  }
  const T dt = (T)A.dt;
  const T bscale = stage == 4 ? dt * (T)(1.0 / 6.0) : (T)1;
  const C* bsrc = reinterpret_cast<const C*>(stage == 4 ? A.lam : A.b_in);
  const int wn = wi.win_hi - wi.win_lo;
  if (sd.has_r && !wi.gread)
    for (int i = tid; i < wn; i += blockDim.x) bw[i] = cscale(bsrc[sd.off_r + wi.win_lo + i], bscale);
  // b_R at flat index i of the system: the staged window, or global memory (scaled on the
  // fly) for tiles without a window
  const C* brg = bsrc + (sd.has_r ? sd.off_r : 0);
  auto b_at = [&](int i) { return wi.gread ? cscale(brg[i], bscale) : bw[i - wi.win_lo]; };
  C* bgx = bw + wn;
  C* bgy = bgx + sd.n_g;
  C* vw = bgy + sd.n_g;  // [nS][2][n_g] source reductions of this system
  const bool do_sep = sd.has_sep && wi.sep_hi > wi.sep_lo;
  if (do_sep) {
    for (int i = tid; i < sd.n_g; i += blockDim.x) {
      bgx[i] = cscale(bsrc[sd.off_gx + i], bscale);
      bgy[i] = cscale(bsrc[sd.off_gy + i], bscale);
    }
  }
  __syncthreads();
  if (do_sep && sd.has_r) {
    const C* srcr = reinterpret_cast<const C*>(A.srcred) + (int64_t)wi.sys * A.srcred_stride;
    for (int i = tid; i < 2 * s_nS * sd.n_g; i += blockDim.x) vw[i] = srcr[i];
  }
  __syncthreads();

  const T* W = reinterpret_cast<const T*>(A.wtab);
  const C* D = reinterpret_cast<const C*>(A.diag) + sd.diag_off;
  const C* U = reinterpret_cast<const C*>(A.u);
  const C* LAM = reinterpret_cast<const C*>(A.lam);
  C* LACC = reinterpret_cast<C*>(A.lacc);
  C* BOUT = reinterpret_cast<C*>(A.b_out);
  int Md[ND];
#pragma unroll
  for (int d = 0; d < ND; ++d) Md[d] = sd.M[d % NM];
  int doff[ND];
  {
    int o = 0;
#pragma unroll
    for (int d = 0; d < ND; ++d) { doff[d] = o; o += Md[d]; }
  }
  // b_{i-1} = dt beta lam + cq dt q
  const T beta = stage == 4 ? (T)(1.0 / 3.0) : (stage == 3 ? (T)(1.0 / 3.0) : (T)(1.0 / 6.0));
  const T cq = stage == 4 ? dt : dt * (T)0.5;
  const int ngt = s_ngt;

  auto finish = [&](int64_t gi, C q) {
    LACC[gi] = stage == 4 ? cadd(LAM[gi], q) : cadd(LACC[gi], q);
    if (stage > 1) BOUT[gi] = caxpy(cq, q, cscale(LAM[gi], dt * beta));
  };
  auto addg = [&](int t, C ub, C bv, T w) {
    // accumulate u * (W b_src) for gradient term t (g is uniform across the warp: a jump
    // to one register accumulator, not a scan over all of them)
    const int g = gidx[t];
    if (g < 0) return;
    const C v = cmul(ub, cscale(bv, w));
    const double vx = (double)v.x, vy = (double)v.y;
    if (g >= BQ_MAX_GT) {
      add_shared(more + 2 * (g - BQ_MAX_GT), vx, vy);
      return;
    }
    switch (g) {
#define BQ_GACC_CASE(q) case q: gacc[q].x += vx; gacc[q].y += vy; break;
      BQ_GACC_CASE(0) BQ_GACC_CASE(1) BQ_GACC_CASE(2) BQ_GACC_CASE(3) BQ_GACC_CASE(4) BQ_GACC_CASE(5)
      BQ_GACC_CASE(6) BQ_GACC_CASE(7) BQ_GACC_CASE(8) BQ_GACC_CASE(9) BQ_GACC_CASE(10) BQ_GACC_CASE(11)
      BQ_GACC_CASE(12) BQ_GACC_CASE(13) BQ_GACC_CASE(14) BQ_GACC_CASE(15)
#undef BQ_GACC_CASE
      default: break;
    }
  };

  // lanes per point: as in the forward stage kernel, lane `sub` of a group of L takes the
  // terms t = sub, sub + L, ... and keeps its own gradient partial sums
  const int L = A.lanes;
  const int sub = tid & (L - 1);
  const unsigned gmask = L == 1 ? (1u << (tid & 31)) : (((1u << L) - 1u) << ((tid & 31) & ~(L - 1)));
  const int pstride = (int)blockDim.x / L;
  auto group_sum = [&](C k) {
    for (int o = 1; o < L; o <<= 1) {
      k.x += __shfl_xor_sync(gmask, k.x, o);
      k.y += __shfl_xor_sync(gmask, k.y, o);
    }
    return k;
  };

  if (sd.has_r) {
    const int ng = sd.n_g;
    for (int p = wi.start + tid / L; p < wi.start + wi.len; p += pstride) {
      int idx[ND];
      const int kx = sd.r_diag ? p : p / ng;  // diagonal residual layout: point p is (p, p)
      const int ly = sd.r_diag ? p : p - kx * ng;
      {
        int r = kx;
#pragma unroll
        for (int d = NM - 1; d >= 0; --d) { idx[d] = r % Md[d]; r /= Md[d]; }
        r = ly;
#pragma unroll
        for (int d = ND - 1; d >= NM; --d) { idx[d] = r % Md[d]; r /= Md[d]; }
      }
      C q = cmk<C>(0.0, 0.0);
      if (sub == 0) {
        C dg = D[doff[0] + idx[0]];
#pragma unroll
        for (int d = 1; d < ND; ++d) dg = cadd(dg, D[doff[d] + idx[d]]);
        q = cmul(dg, b_at(p));
      }
      const C up = U[sd.off_r + p];
      for (int t = sub; t < nt; t += L) {
        const TermDesc& td = st[t];
        // secular projector term: it shifts x and y alike, so its source p - delta lies on the
        // diagonal of its mode exactly when p does
        if (td.diagp1 && idx[td.diagp1 - 1] != idx[NM + td.diagp1 - 1]) continue;
        // diagonal layout: only terms that shift x and y alike couple diagonal points (the
        // projection D of the forward equation), at offset deltaGx in the diagonal index
        if (sd.r_diag && td.deltaGx != td.deltaGy) continue;
        T w = (T)1;
        bool ok = true;
        for (int i = 0; i < td.n_act; ++i) {
          const int d = td.dim[i];
          const int s = idx[d] - td.sh[i];
          ok = ok && (s >= 0) && (s < Md[d]);
          w *= ok ? W[td.wtab[i] + (ok ? s : 0)] : (T)0;
        }
        if (!ok) w = (T)0;
        const int src = (w != (T)0) ? p - (sd.r_diag ? td.deltaGx : td.deltaR) : p;
        const C bv = b_at(src);
        q = cfma(sc[t], cscale(bv, w), q);
        if (ngt) addg(t, up, bv, w);
      }
      q = group_sum(q);
      if (sub == 0) finish(sd.off_r + p, q);
    }
  }
  if (do_sep) {
    const int ng = sd.n_g;
    const C Cc = cmk<C>(sd.c_re, sd.c_im);
    for (int i = wi.sep_lo + tid / L; i < wi.sep_hi; i += pstride) {
      const int side = i < ng ? SIDE_X : SIDE_Y;
      const int g = side == SIDE_X ? i : i - ng;
      const int d0 = side == SIDE_X ? 0 : NM;
      int idx[ND];
      {
        int r = g;
#pragma unroll
        for (int d = NM - 1; d >= 0; --d) { idx[d0 + d] = r % Md[d]; r /= Md[d]; }
      }
      const C* bs = side == SIDE_X ? bgx : bgy;
      C q = cmk<C>(0.0, 0.0);
      const C up = U[(side == SIDE_X ? sd.off_gx : sd.off_gy) + g];
      if (sub == 0) {
        C dg = side == SIDE_X ? Cc : cmk<C>(-sd.c_re, -sd.c_im);
#pragma unroll
        for (int d = 0; d < NM; ++d) dg = cadd(dg, D[doff[d0 + d] + idx[d0 + d]]);
        q = cmul(dg, bs[g]);
        const C v = cmul(up, bs[g]);
        if (side == SIDE_X) { dcacc.x += (double)v.x; dcacc.y += (double)v.y; }
        else { dcacc.x -= (double)v.x; dcacc.y -= (double)v.y; }
      }
      for (int t = sub; t < nt; t += L) {
        const TermDesc& td = st[t];
        const bool own = td.side == side;
        const bool src_term = td.side == SIDE_S && sd.has_r;
        if (!own && !src_term) continue;
        // weight over the active dims of this side
        T w = (T)1;
        bool ok = true;
        for (int j = 0; j < td.n_act; ++j) {
          const int d = td.dim[j];
          if ((d < NM) != (side == SIDE_X)) continue;
          const int s = idx[d] - td.sh[j];
          ok = ok && (s >= 0) && (s < Md[d]);
          w *= ok ? W[td.wtab[j] + (ok ? s : 0)] : (T)0;
        }
        if (!ok) w = (T)0;
        const int delta = side == SIDE_X ? td.deltaGx : td.deltaGy;
        const int src = (w != (T)0) ? g - delta : g;
        if (own) {
          const C bv = bs[src];
          q = cfma(sc[t], cscale(bv, w), q);
          if (ngt) addg(t, up, bv, w);
        } else {
          // d/dG_x of  c (Wx G_x[.+sx]) (Wy G_y[.+sy]) paired with b_R: c Wx(j-sx) v_t[j-sx]
          const C* red_t = vw + (sidx[t] * 2 + (side == SIDE_X ? 0 : 1)) * ng;
          q = cfma(sc[t], cscale(red_t[src], w), q);
        }
      }
      q = group_sum(q);
      if (sub == 0) finish((side == SIDE_X ? sd.off_gx : sd.off_gy) + g, q);
    }
  }

  // ---- gradient reductions: per-warp reduce-scatter, then one atomic per term per CTA --
  // The 2 BQ_MAX_GT = 32 real partial sums of every lane are reduced across the warp by
  // halving exchanges (at offset o a lane keeps the half of its values selected by bit o of
  // its lane index and adds the partner's copy of that half): 31 additions per lane instead
  // of 5 per value, and afterwards lane j holds the warp's sum of value j.
  static_assert(2 * BQ_MAX_GT == 32, "the reduce-scatter maps one value to each lane");
  if (accumulate && !last) {
    // keep the partial sums unless a gradient term's factor changes before the next call
    // (uniform over the CTA: it depends on the terms and the times only)
    bool change = false;
    for (int t = 0; t < nt && !change; ++t) {
      if (gidx[t] < 0 || st[t].ch < 0) continue;
      const ChanDesc cd = A.chans[st[t].ch];
      if (cd.kind == 0) continue;  // constant
      if (cd.kind != 2) { change = true; break; }
      if (stage == 1) {  // the next call is the previous step: its piecewise-constant segment
        const double tm = A.tau_step + 0.5 * A.dt, tn = tm - A.dt;
        const int s0 = pwc_segment(cd, A.chpar, A.reverse ? A.horizon - tm : tm);
        const int s1 = pwc_segment(cd, A.chpar, A.reverse ? A.horizon - tn : tn);
        change = s0 != s1;
      }
    }
    if (!change) return;
  }
  if (ngt > 0 || (do_sep && sd.n_params > 0)) {
    const int lane = tid & 31, warp = tid >> 5;
    double v[32];
#pragma unroll
    for (int g = 0; g < BQ_MAX_GT; ++g) { v[2 * g] = gacc[g].x; v[2 * g + 1] = gacc[g].y; }
#pragma unroll
    for (int lev = 0; lev < 5; ++lev) {
      const int o = 16 >> lev, h = 16 >> lev;  // h values kept out of 2 h
      const bool upper = (lane & o) != 0;
#pragma unroll
      for (int j = 0; j < h; ++j) {
        const double send = upper ? v[j] : v[j + h];
        const double keep = upper ? v[j + h] : v[j];
        v[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    }
    red[warp][lane] = v[0];
    double2 dv = dcacc;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      dv.x += __shfl_down_sync(0xffffffffu, dv.x, o);
      dv.y += __shfl_down_sync(0xffffffffu, dv.y, o);
    }
    if (lane == 0) { red[warp][32] = dv.x; red[warp][33] = dv.y; }
    __syncthreads();
    if (tid < nt) {
      const int t = tid;
      const int g = gidx[t];
      if (g >= 0) {
        double2 a = make_double2(0.0, 0.0);
        if (g < BQ_MAX_GT) {
          for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { a.x += red[w][2 * g]; a.y += red[w][2 * g + 1]; }
        } else {
          double* m = more + 2 * (g - BQ_MAX_GT);
          a = make_double2(m[0], m[1]);
          m[0] = m[1] = 0.0;
        }
        const TermDesc& td = st[t];
        double2 e = make_double2(1.0, 0.0);
        double t_phys = 0.0;
        if (td.ch >= 0) {
          const ChanDesc cd = A.chans[td.ch];
          const double tau = (cd.kind == 2) ? A.tau_step + 0.5 * A.dt : A.tau_step + stage_c(stage) * A.dt;
          t_phys = A.reverse ? A.horizon - tau : tau;
          e = chan_value(cd, A.chpar, t_phys);
          if (td.conj) e.y = -e.y;
        }
        if (td.gslot_param >= 0) {
          // d coef / d theta = cb * channel
          const double cr = td.cb_re * e.x - td.cb_im * e.y, ci = td.cb_re * e.y + td.cb_im * e.x;
          atomicAdd(A.grad + td.gslot_param, cr * a.x - ci * a.y);
        }
        if (td.gslot_pwc >= 0) {
          const ChanDesc cd = A.chans[td.ch];
          const int sg = pwc_segment(cd, A.chpar, t_phys);
          if (sg >= 0) {
            // d/dRe: c; d/dIm: +i c (channel) or -i c (conjugate channel)
            const double re = td.c_re * a.x - td.c_im * a.y;
            const double im = td.c_re * a.y + td.c_im * a.x;
            atomicAdd(A.grad + td.gslot_pwc + 2 * sg, re);
            atomicAdd(A.grad + td.gslot_pwc + 2 * sg + 1, td.conj ? im : -im);
          }
        }
      }
    }
    if (do_sep && tid < sd.n_params) {
      double2 a = make_double2(0.0, 0.0);
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { a.x += red[w][32]; a.y += red[w][33]; }
      const double2 dcv = A.dc[sd.dc_off + tid];
      atomicAdd(A.grad + sd.grad_off + tid, dcv.x * a.x - dcv.y * a.y);
    }
  }
#pragma unroll
  for (int g = 0; g < BQ_MAX_GT; ++g) gacc[g] = make_double2(0.0, 0.0);
  dcacc = make_double2(0.0, 0.0);
}

template <typename T, int NM>
__global__ void __launch_bounds__(BQ_BLOCK) k_adj_stage(const AdjArgs A) {
  double2 gacc[BQ_MAX_GT];
#pragma unroll
  for (int g = 0; g < BQ_MAX_GT; ++g) gacc[g] = make_double2(0.0, 0.0);
  double2 dcacc = make_double2(0.0, 0.0);
  adj_stage_body<T, NM>(A, blockIdx.x, true, gacc, dcacc, false, true);
}

// Transposed separable source: for every system and sandwich term t
//   v_t[kx] = sum_ly b_R[kx, ly] Wy_t(ly) G_y[ly + sy],   w_t[ly] = sum_kx b_R[kx, ly] Wx_t(kx) G_x[kx + sx]
// (G_x, G_y of the recorded stage input; b_R = dt/6 lam at stage 4).  grid = (systems, max S terms, 2).
#define BQ_SRC_THREADS 256
#define BQ_SRC_TILE 8      // outputs per CTA (one row per warp; BQ_SRC_THREADS / 8 partial sums per column)
// outputs per CTA in the cooperative backward kernel (BQ_BLOCK threads): smaller tiles give the
// phase more items, since the CTAs of a cooperative launch that have none just wait
#define BQ_SRC_TILE_COOP 4
#define BQ_SRC_ZCH 1024    // summed-index chunk held in shared memory
// One CTA's part of the transposed source, (bx, by, bz) = (system, sandwich term, direction
// and output tile), with NTH threads (k_adj_src: BQ_SRC_THREADS; the cooperative backward
// segment kernel: BQ_BLOCK).
template <typename T, int NM, int NTH, int TILE>
__device__ __forceinline__ void adj_src_body(const AdjArgs& A, int bx, int by, int bz) {
  static_assert(TILE % (NTH / 32) == 0, "every warp sums TILE / (NTH / 32) rows");
  using C = typename C2T<T>::type;
  __shared__ C z[BQ_SRC_ZCH];
  __shared__ C red[NTH / TILE][TILE];
  __syncthreads();  // the CTA's previous item is done with z and red
  const SysDesc& sd = A.sys[bx];
  if (!sd.has_sep || !sd.has_r) return;
  // the by-th sandwich term of the system
  int t = -1, s = 0;
  for (int q = 0; q < sd.n_terms; ++q)
    if (A.terms[sd.term_off + q].side == SIDE_S) {
      if (s == by) { t = q; break; }
      ++s;
    }
  if (t < 0) return;
  const TermDesc td = A.terms[sd.term_off + t];
  const int dirx = (bz & 1) == 0;  // 1: v_t over kx (sum over ly), 0: w_t over ly (sum over kx)
  const int i0 = (bz >> 1) * TILE;
  const int ng = sd.n_g;
  if (i0 >= ng) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const T dt = (T)A.dt;
  const T bscale = A.stage == 4 ? dt * (T)(1.0 / 6.0) : (T)1;
  const C* bsrc = reinterpret_cast<const C*>(A.stage == 4 ? A.lam : A.b_in) + sd.off_r;
  const C* U = reinterpret_cast<const C*>(A.u);
  const C* other = U + (dirx ? sd.off_gy : sd.off_gx);
  const T* W = reinterpret_cast<const T*>(A.wtab);
  const int delta = dirx ? td.deltaGy : td.deltaGx;
  // secular projector term: only pairs whose indices of mode dm agree contribute
  const int dm = td.diagp1 - 1;
  auto midx = [&](int f) { return dm >= 0 ? (f / sd.stG[dm]) % sd.M[dm] : 0; };
  if (sd.r_diag) {
    // diagonal layout: B(i, j) is zero off i = j, so out[i] = bscale b_R[i] z[i]
    if (tid < TILE && i0 + tid < ng) {
      const int i = i0 + tid;
      int rem = i;
      int id[NM];
#pragma unroll
      for (int d = NM - 1; d >= 0; --d) { id[d] = rem % sd.M[d]; rem /= sd.M[d]; }
      T w = (T)1;
      for (int a = 0; a < td.n_act; ++a) {
        const int d = td.dim[a];
        const bool isx = d < NM;
        if (isx == (bool)dirx) continue;  // the summed side's dims
        w *= W[td.wtab[a] + id[isx ? d : d - NM]];
      }
      const C zi = w == (T)0 ? cmk<C>(0.0, 0.0) : cscale(other[i + delta], w);
      C* outd = reinterpret_cast<C*>(const_cast<void*>(A.srcred)) + (int64_t)bx * A.srcred_stride +
                (s * 2 + (dirx ? 0 : 1)) * ng;
      outd[i] = cscale(cmul(bsrc[i], zi), bscale);
    }
    return;
  }
  // out[i] = bscale sum_j B(i, j) z[j], z[j] = w(j) other[j + delta], with B(i, j) the R
  // cotangent at (i, j) (dirx) or (j, i), and w(j) the product of the term's weights on the
  // summed side.  Chunks of z go through shared memory; the sums run in a fixed order.
  C acc[TILE / (NTH / 32)];
#pragma unroll
  for (int r = 0; r < TILE / (NTH / 32); ++r) acc[r] = cmk<C>(0.0, 0.0);
  C accc = cmk<C>(0.0, 0.0);
  for (int jc = 0; jc < ng; jc += BQ_SRC_ZCH) {
    const int nj = min(BQ_SRC_ZCH, ng - jc);
    __syncthreads();  // the previous chunk is consumed
    for (int jj = tid; jj < nj; jj += NTH) {
      const int j = jc + jj;
      int rem = j;
      int id[NM];
#pragma unroll
      for (int d = NM - 1; d >= 0; --d) { id[d] = rem % sd.M[d]; rem /= sd.M[d]; }
      T w = (T)1;
      for (int a = 0; a < td.n_act; ++a) {
        const int d = td.dim[a];
        const bool isx = d < NM;
        if (isx == (bool)dirx) continue;  // only the summed side's dims
        w *= W[td.wtab[a] + id[isx ? d : d - NM]];
      }
      z[jj] = w == (T)0 ? cmk<C>(0.0, 0.0) : cscale(other[j + delta], w);
    }
    __syncthreads();
    if (dirx) {
      // rows i0 + warp * R + r: lanes stride over j (coalesced along the row)
#pragma unroll
      for (int r = 0; r < TILE / (NTH / 32); ++r) {
        const int i = i0 + warp * (TILE / (NTH / 32)) + r;
        if (i < ng) {
          const C* row = bsrc + (int64_t)i * ng + jc;
          const int mi = midx(i);
          for (int jj = lane; jj < nj; jj += 32)
            if (dm < 0 || midx(jc + jj) == mi) acc[r] = cfma(row[jj], z[jj], acc[r]);
        }
      }
    } else {
      // column i0 + tid % TILE: the CTA's NTH / TILE thread groups split j (each
      // group reads TILE adjacent columns of one row)
      const int i = i0 + tid % TILE;
      const int mi = midx(i);
      if (i < ng)
        for (int jj = tid / TILE; jj < nj; jj += NTH / TILE)
          if (dm < 0 || midx(jc + jj) == mi) accc = cfma(bsrc[(int64_t)(jc + jj) * ng + i], z[jj], accc);
    }
  }
  C* out = reinterpret_cast<C*>(const_cast<void*>(A.srcred)) + (int64_t)bx * A.srcred_stride +
           (s * 2 + (dirx ? 0 : 1)) * ng;
  if (dirx) {
#pragma unroll
    for (int r = 0; r < TILE / (NTH / 32); ++r) {
      C v = acc[r];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_down_sync(0xffffffffu, v.x, o);
        v.y += __shfl_down_sync(0xffffffffu, v.y, o);
      }
      const int i = i0 + warp * (TILE / (NTH / 32)) + r;
      if (lane == 0 && i < ng) out[i] = cscale(v, bscale);
    }
  } else {
    red[tid / TILE][tid % TILE] = accc;
    __syncthreads();
    if (tid < TILE) {
      C v = red[0][tid];
      for (int w2 = 1; w2 < NTH / TILE; ++w2) v = cadd(v, red[w2][tid]);
      const int i = i0 + tid;
      if (i < ng) out[i] = cscale(v, bscale);
    }
  }
}

template <typename T, int NM>
__global__ void __launch_bounds__(BQ_SRC_THREADS) k_adj_src(const AdjArgs A) {
  adj_src_body<T, NM, BQ_SRC_THREADS, BQ_SRC_TILE>(A, blockIdx.x, blockIdx.y, blockIdx.z);
}

// ---------------------------------------------------------------------------------------
// Cooperative segment kernels of the gradient.  A checkpoint segment of a small state is a
// long chain of short dependent stages; one launch per stage leaves the GPU mostly idle
// between them.  Here one cooperative launch (every CTA resident, so the CTAs can wait for
// one another) runs all stages of a segment: each CTA takes the work items blockIdx.x,
// blockIdx.x + gridDim.x, ... of a phase, and a grid barrier separates dependent phases.
// With at most one item per CTA the item's descriptors stay in shared memory for the whole
// segment.
// ---------------------------------------------------------------------------------------
#define BQ_GRID_WAIT_CYCLES (4000000000LL)  // about 2 s at the maximum SM clock

// Grid-wide barrier of a cooperative launch: thread 0 of each CTA arrives (release) and waits
// (acquire) for the generation to change; the last arrival resets the count and starts the
// next generation.  The wait is bounded: on timeout the CTA sets bit 2 of *error and the
// caller returns (the other CTAs then time out at the same barrier or the next).
__device__ __forceinline__ bool grid_barrier(unsigned int* bar, unsigned int* error) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned int gen;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(gen) : "l"(bar + 1) : "memory");
    unsigned int old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(bar) : "memory");
    int ok = 1;
    if (old == gridDim.x - 1) {
      asm volatile("st.relaxed.gpu.global.u32 [%0], 0;" ::"l"(bar) : "memory");
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar + 1) : "memory");
    } else {
      const long long t0 = clock64();
      for (;;) {
        unsigned int g;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(g) : "l"(bar + 1) : "memory");
        if (g != gen) break;
        if (clock64() - t0 > BQ_GRID_WAIT_CYCLES) {
          ok = 0;
          atomicOr(error, 4u);
          break;
        }
        __nanosleep(40);
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// Forward stages of n_steps steps from y (and comp), the stage inputs alternating between ua
// and ub as in the per-stage launches; with rec, every stage input is also recorded at
// rec + (4 i + stage - 1) arr.
template <typename T, int NM>
__global__ void __launch_bounds__(BQ_BLOCK) k_coop_fwd(const CoopArgs P) {
  const bool reload = P.n_work > (int)gridDim.x;
  bool first = true;
  for (int i = 0; i < P.n_steps; ++i) {
    const double tau = P.tau0 + (double)i * P.st.dt;
    for (int stage = 1; stage <= 4; ++stage) {
      StageArgs a = P.st;
      a.stage = stage;
      a.u_in = stage == 1 ? a.y : (stage == 2 ? P.ua : (stage == 3 ? P.ub : P.ua));
      a.u_out = stage == 1 ? P.ua : (stage == 2 ? P.ub : (stage == 3 ? P.ua : nullptr));
      a.rec = P.rec ? P.rec + ((size_t)i * 4 + stage - 1) * P.arr : nullptr;
      for (int it = blockIdx.x; it < P.n_work; it += gridDim.x) {
        stage_body<T, NM>(a, it, tau, reload || first);
        first = false;
      }
      if (!grid_barrier(P.bar, P.error)) return;
    }
  }
}

// Adjoint of the segment's steps, last step first, from the recorded stage inputs: per stage
// the transposed-source reductions (if the systems have sandwich terms), a barrier, the
// transposed stage with the parameter gradients, a barrier.  lam and lacc swap after every
// step, as in the per-stage launches; the cotangent before the segment ends in lam if
// n_steps is even, else in lacc.
template <typename T, int NM>
__global__ void __launch_bounds__(BQ_BLOCK) k_coop_bwd(const CoopArgs P) {
  const bool reload = P.n_work > (int)gridDim.x;
  bool first = true;
  // per-thread partial gradient sums, kept across the stages of the segment when every CTA
  // keeps one item (reduced into the gradient slots when a factor changes and at the end)
  double2 gacc[BQ_MAX_GT];
#pragma unroll
  for (int g = 0; g < BQ_MAX_GT; ++g) gacc[g] = make_double2(0.0, 0.0);
  double2 dcacc = make_double2(0.0, 0.0);
  void* lam = P.lam;
  void* lacc = P.lacc;
  const int src_per_sys = P.max_s * 2 * P.src_tiles;
  const int n_src = P.max_s > 0 ? P.n_sys * src_per_sys : 0;
  for (int n = P.n_steps - 1; n >= 0; --n) {
    for (int stage = 4; stage >= 1; --stage) {
      AdjArgs a = P.adj;
      a.stage = stage;
      a.tau_step = P.tau0 + (double)n * a.dt;
      a.lam = lam;
      a.lacc = lacc;
      a.u = P.rec + ((size_t)n * 4 + stage - 1) * P.arr;
      a.b_in = stage == 4 ? nullptr : (stage == 3 ? P.ba : (stage == 2 ? P.bb : P.ba));
      a.b_out = stage == 4 ? P.ba : (stage == 3 ? P.bb : (stage == 2 ? P.ba : nullptr));
      if (n_src > 0) {
        for (int it = blockIdx.x; it < n_src; it += gridDim.x) {
          const int bx = it / src_per_sys, rem = it - bx * src_per_sys;
          adj_src_body<T, NM, BQ_BLOCK, BQ_SRC_TILE_COOP>(a, bx, rem / (2 * P.src_tiles), rem % (2 * P.src_tiles));
        }
        if (!grid_barrier(P.bar, P.error)) return;
      }
      for (int it = blockIdx.x; it < P.n_work; it += gridDim.x) {
        adj_stage_body<T, NM>(a, it, reload || first, gacc, dcacc, !reload, n == 0 && stage == 1);
        first = false;
      }
      if (!grid_barrier(P.bar, P.error)) return;
    }
    void* t = lam;
    lam = lacc;
    lacc = t;
  }
}

// Cotangent of the final state for l = Re sum_b Tr(rho0_b A_b): one thread per system.
template <typename T>
__global__ void k_adj_seed(const SysDesc* __restrict__ sys, const EvalGroup* __restrict__ groups,
                           const EvalEntry* __restrict__ entries, const void* ystate, void* lam, int n_groups) {
  using C = typename C2T<T>::type;
  const int gi = blockIdx.x * blockDim.x + threadIdx.x;
  if (gi >= n_groups) return;
  const EvalGroup g = groups[gi];
  const C* y = reinterpret_cast<const C*>(ystate);
  C* L = reinterpret_cast<C*>(lam);
  for (int s = 0; s < g.n_sys; ++s) {
    const SysDesc& sd = sys[g.sys_off + s];
    for (int e = 0; e < g.n_e; ++e) {
      const EvalEntry en = entries[g.e_off + e];
      const double fr = sd.w_re * en.f_re - sd.w_im * en.f_im;
      const double fi = sd.w_re * en.f_im + sd.w_im * en.f_re;
      const C f = cmk<C>(fr, fi);
      if (sd.has_r && (!sd.r_diag || en.kx == en.ly)) {  // the diagonal layout keeps k = l only
        C& r = L[sd.off_r + (sd.r_diag ? (int64_t)en.kx : (int64_t)en.kx * sd.n_g + en.ly)];
        r = cadd(r, f);
      }
      if (sd.has_sep) {
        C& ax = L[sd.off_gx + en.kx];
        C& ay = L[sd.off_gy + en.ly];
        const C gx = y[sd.off_gx + en.kx];
        const C gy = y[sd.off_gy + en.ly];
        ax = cfma(f, gy, ax);
        ay = cfma(f, gx, ay);
      }
    }
  }
}

// ---------------------------------------------------------------------------------------
// Batched persistent solve, merged-stencil form (single mode, every shift in {-1, 0, 1}):
// the solve of k_solve_m1 with the per-term stencil replaced by per-row / per-column
// coefficient vectors (rebuilt for the next stage while the current one is computed) and a
// column-strip thread mapping with a register window of the stage input.  Thread (l, b)
// owns column l, rows [b rb, (b+1) rb) (rb even: two rows per iteration); the state y of its
// points stays in registers, their stage sum and compensation in shared memory, for the
// whole solve (FP32: 80 registers, three CTAs per SM).  One barrier per stage; coefficients
// are evaluated two stages ahead (triple buffered), the merged vectors one stage ahead
// (double buffered), each role in warps of its own.
// ---------------------------------------------------------------------------------------
template <typename T, int BLK, int RB, int MX, int MY, int MS, bool DIAG>
__global__ void __launch_bounds__(BLK, sizeof(T) == 4 ? 3 : 1) k_solve_mg(const SolveArgs A) {
  using C = typename C2T<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ M1Sys s;
  __shared__ C coef[3][3 * BQ_M1_MAXT];
  __shared__ float cf32[3 * BQ_M1_MAXT][8];  // FP32 stage coefficients (see eval_coef)
  __shared__ float tp32[4];                  // t0 and dt as FP32 pairs (hi, lo)
  __shared__ int s_next;
  const int tid = threadIdx.x;
  C* y_g = reinterpret_cast<C*>(A.y);
  C* comp_g = reinterpret_cast<C*>(A.comp);
  const C zero = cmk<C>(0.0, 0.0);

  for (;;) {
    if (tid == 0) s_next = (int)atomicAdd(A.queue, 1u);
    __syncthreads();
    const int qi = s_next;
    if (qi >= A.n_sys) return;
    {
      const int* src = reinterpret_cast<const int*>(A.m1 + A.order[qi]);
      int* dst = reinterpret_cast<int*>(&s);
      for (int i = tid; i < (int)(sizeof(M1Sys) / sizeof(int)); i += BLK) dst[i] = src[i];
    }
    __syncthreads();
    const int M = s.M, nX = s.nX, nY = s.nY, nS = s.nS;
    const int sdiag = s.sdiag;  // bit q: sandwich term q acts only where k = l
    const int has_r = s.has_r, has_sep = s.has_sep;
    const int nr = has_r ? M * M : 0;
    const int ntot = nr + (has_sep ? 2 * M : 0);
    // shared: B0[ntot] | B1[ntot] | AS[nr] CS[nr] | dx[M] dy[M] | MV[2][(6 + MS) M] | wX wY wSx
    // wSy (real).  AS and CS hold the stage sum and the compensation of the R points (each
    // touched only by the thread that owns the point; in shared memory rather than registers,
    // so that three CTAs fit an SM in FP32)
    C* B0 = reinterpret_cast<C*>(smem_raw);
    C* B1 = B0 + ntot;
    C* AS = B1 + ntot;
    C* CS = AS + nr;
    C* dx = CS + nr;
    C* dy = dx + M;
    C* MV = dy + M;
    const int mvs = (6 + MS) * M;
    T* wX = reinterpret_cast<T*>(MV + 2 * mvs);
    T* wY = wX + nX * M;
    T* wSx = wY + nY * M;
    T* wSy = wSx + nS * M;
    const int nt = nX + nY + nS;
    // Thread roles besides the strips, each in warps of its own counted from the top of the
    // block down, so that no warp carries more than one of them on top of its strip (a warp
    // runs its lanes' roles one after the other, and the slowest warp sets every stage's
    // barrier): the G items (the last 2M threads), the column entries of the merged vectors,
    // their row entries, the stage coefficients.  With M <= 42 and at most 10 terms (4 X,
    // 4 Y, 2 sandwich) they fit below the block's top without overlap (BLK = 256).
    const int g_lo = BLK - (has_sep ? 2 * M : 0);
    const int bc_lo = max((g_lo & ~31) - M, 0);
    const int br_lo = max((bc_lo & ~31) - M, 0);
    const int c_lo = max((br_lo & ~31) - nt, 0);
    // Stage coefficient c_t e(t) of term t.  In FP64, and in FP32 for envelopes other than a
    // Gaussian: the stage time in FP64, the envelope and the product in the state's precision.
    // An FP32 Gaussian costs no FP64 operation (this sits on a warp's path every stage, and
    // GB300's FP64 rate is a small fraction of its FP32 rate): its amplitude, 1 / (2 sigma^2)
    // and centre (an FP32 pair) are set once per system in cf32; the stage time t = t0 + x dt
    // (x = step + c_s, exact in FP32 below 2^23 steps; reversed reading: t0 = horizon - tau0
    // and -dt) is formed as an unevaluated FP32 pair from the pairs of t0 and dt (error-free
    // product by FMA, TwoSum), and t - centre = (t_hi - c_hi) + (t_lo - c_lo) is exact to the
    // rounding of the difference wherever the pulse is not negligible.
    auto eval_coef = [&](int buf, int64_t step, int stage) {
      const int ct = tid - c_lo;
      if (ct >= 0 && ct < nt) {
        const float* k = cf32[ct];
        if (sizeof(T) == 4 && k[2] > 0.5f) {
          const float x = (float)step + (stage == 1 ? 0.f : (stage == 4 ? 1.f : 0.5f));
          const float ph = x * tp32[2];
          const float pl = fmaf(x, tp32[2], -ph) + x * tp32[3];
          const float th = tp32[0] + ph;
          const float bv = th - tp32[0];
          const float tl = ((tp32[0] - (th - bv)) + (ph - bv)) + (tp32[1] + pl);
          const float d = (th - k[6]) + (tl - k[7]);
          const float g = dev_exp<float>(-(d * d) * k[5]);
          coef[buf][ct] = cmul(cmk<C>(k[0], k[1]), cmk<C>(k[3] * g, k[4] * g));
          return;
        }
        const int t = ct < nX ? s.tX[ct] : (ct < nX + nY ? s.tY[ct - nX] : s.tS[ct - nX - nY]);
        const TermDesc& td = A.terms[s.term_off + t];
        C c = cmk<C>(td.c_re, td.c_im);
        if (td.ch >= 0) {
          const ChanDesc cd = A.chans[td.ch];
          const double ts = A.tau0 + (double)step * A.dt;
          const double tau = (cd.kind == 2) ? ts + 0.5 * A.dt : ts + stage_c(stage) * A.dt;
          const double2 e = chan_value_t<T>(cd, A.chpar, A.reverse ? A.horizon - tau : tau);
          c = cmul(c, cmk<C>(e.x, td.conj ? -e.y : e.y));
        }
        coef[buf][ct] = c;
      }
    };
    {
      const int ct = tid - c_lo;
      if (ct >= 0 && ct < nt) {
        float* k = cf32[ct];
        k[2] = 0.f;
        if (sizeof(T) == 4 && A.n_steps < (1LL << 23)) {
          const int t = ct < nX ? s.tX[ct] : (ct < nX + nY ? s.tY[ct - nX] : s.tS[ct - nX - nY]);
          const TermDesc& td = A.terms[s.term_off + t];
          if (td.ch >= 0 && A.chans[td.ch].kind == 1) {
            const double* p = A.chpar + A.chans[td.ch].par_off;
            k[0] = (float)td.c_re;
            k[1] = (float)td.c_im;
            k[2] = 1.f;
            k[3] = (float)p[0];
            k[4] = (float)(td.conj ? -p[1] : p[1]);
            k[5] = (float)(1.0 / (2.0 * p[3] * p[3]));
            k[6] = (float)p[2];
            k[7] = (float)(p[2] - (double)k[6]);
          }
        }
      }
      if (tid == c_lo) {
        const double t0 = A.reverse ? A.horizon - A.tau0 : A.tau0;
        const double d0 = A.reverse ? -A.dt : A.dt;
        tp32[0] = (float)t0;
        tp32[1] = (float)(t0 - (double)tp32[0]);
        tp32[2] = (float)d0;
        tp32[3] = (float)(d0 - (double)tp32[2]);
      }
      __syncthreads();
    }
    // merged vectors from coef[cb] into MV half mb: A0 Am Ap (rows) B0 Bm Bp (columns) SX_t
    auto build_mv = [&](int cb, int mb) {
      C* V = MV + mb * mvs;
      if (tid >= br_lo && tid < br_lo + M) {  // row i: A0, Am, Ap and the sandwich rows
        const int i = tid - br_lo;
        C a0 = dx[i], am = zero, ap = zero;
#pragma unroll
        for (int q = 0; q < MX; ++q)
          if (q < nX) {
            const C v = cscale(coef[cb][q], wX[q * M + i]);
            if (s.sX[q] == 0) a0 = cadd(a0, v); else if (s.sX[q] < 0) am = cadd(am, v); else ap = cadd(ap, v);
          }
        V[i] = a0; V[M + i] = am; V[2 * M + i] = ap;
#pragma unroll
        for (int q = 0; q < MS; ++q)
          if (q < nS) V[(6 + q) * M + i] = cscale(coef[cb][nX + nY + q], wSx[q * M + i]);
      } else if (tid >= bc_lo && tid < bc_lo + M) {  // column i: B0, Bm, Bp
        const int i = tid - bc_lo;
        C b0 = dy[i], bm = zero, bp = zero;
#pragma unroll
        for (int q = 0; q < MY; ++q)
          if (q < nY) {
            const C v = cscale(coef[cb][nX + q], wY[q * M + i]);
            if (s.sY[q] == 0) b0 = cadd(b0, v); else if (s.sY[q] < 0) bm = cadd(bm, v); else bp = cadd(bp, v);
          }
        V[3 * M + i] = b0; V[4 * M + i] = bm; V[5 * M + i] = bp;
      }
    };
    // ---- load: state, tables; coefficients of stages (0,1) and (0,2); vectors of (0,1) ----
    // column strips of rb rows, rb even (the strip loop takes two rows per iteration): nb
    // strips of the M columns' np = ceil(M / 2) row pairs
    const int np = (M + 1) / 2;
    const int nb = min(BLK / M, np);
    const int rb = 2 * ((np + nb - 1) / nb);
    const int cl = tid % M, cbk = tid / M;
    const bool owner = has_r && cbk < nb;
    const int k0 = cbk * rb, k1 = owner ? min(M, k0 + rb) : k0;
    C yv[RB];
    auto gidx_r = [&](int kk) { return s.off_r + (int64_t)kk * M + cl; };
#pragma unroll
    for (int j = 0; j < RB; ++j) {
      const int kk = k0 + j;
      if (kk < k1) {
        yv[j] = y_g[gidx_r(kk)];
        CS[kk * M + cl] = comp_g[gidx_r(kk)];
        B0[kk * M + cl] = yv[j];
      } else {
        yv[j] = zero;
      }
    }
    // G_x, G_y (elements nr .. nr + 2M): thread g_lo + q owns element nr + q
    const bool gown = has_sep && tid >= g_lo;
    const int gq = tid - g_lo;
    C gy_v = zero, ga_v = zero, gc_v = zero;
    const int64_t g_gi = gown ? (gq < M ? s.off_gx + gq : s.off_gy + (gq - M)) : 0;
    if (gown) {
      gy_v = y_g[g_gi];
      gc_v = comp_g[g_gi];
      B0[nr + gq] = gy_v;
    }
    {
      const C* Dg = reinterpret_cast<const C*>(A.diag) + s.diag_off;
      const T* W = reinterpret_cast<const T*>(A.wtab);
      for (int i = tid; i < M; i += BLK) {
        dx[i] = Dg[i];
        dy[i] = Dg[M + i];
#pragma unroll
        for (int j = 0; j < MX; ++j) if (j < nX) wX[j * M + i] = s.wX[j] >= 0 ? W[s.wX[j] + i] : (T)1;
#pragma unroll
        for (int j = 0; j < MY; ++j) if (j < nY) wY[j * M + i] = s.wY[j] >= 0 ? W[s.wY[j] + i] : (T)1;
#pragma unroll
        for (int j = 0; j < MS; ++j)
          if (j < nS) {
            wSx[j * M + i] = s.wSx[j] >= 0 ? W[s.wSx[j] + i] : (T)1;
            wSy[j * M + i] = s.wSy[j] >= 0 ? W[s.wSy[j] + i] : (T)1;
          }
      }
    }
    eval_coef(0, 0, 1);
    eval_coef(1, 0, 2);
    __syncthreads();
    build_mv(0, 0);
    __syncthreads();
    const C Cc = cmk<C>(s.c_re, s.c_im);
    const C mCc = cmk<C>(-s.c_re, -s.c_im);
    const T dt = (T)A.dt;
    int ssx[MS], ssy[MS];
#pragma unroll
    for (int q = 0; q < MS; ++q) { ssx[q] = s.sSx[q]; ssy[q] = s.sSy[q]; }

    int cbuf = 0;  // coef buffer of the current stage; +1 (mod 3) is the next stage's
    int mbuf = 0;  // MV half of the current stage
    for (int64_t step = 0; step < A.n_steps; ++step) {
#pragma unroll 1
      for (int stage = 1; stage <= 4; ++stage) {
        const C* uin = (stage & 1) ? B0 : B1;
        C* uout = (stage & 1) ? B1 : B0;
        const C* V = MV + mbuf * mvs;
        const C* gxi = uin + nr;
        const C* gyi = gxi + M;
        // coefficients two stages ahead (stage + 2)
        {
          int st2 = stage + 2;
          int64_t sp2 = step;
          if (st2 > 4) { st2 -= 4; ++sp2; }
          eval_coef((cbuf + 2) % 3, sp2, st2);
        }
        if (owner) {
          const C b0 = V[3 * M + cl], bm = V[4 * M + cl], bp = V[5 * M + cl];
          T sy[MS];
          C gyp[MS];
#pragma unroll
          for (int q = 0; q < MS; ++q) {
            sy[q] = q < nS ? wSy[q * M + cl] : (T)0;
            const int yy = cl + ssy[q];
            gyp[q] = (q < nS && has_sep && yy >= 0 && yy < M) ? cscale(gyi[yy], sy[q]) : zero;
          }
          const bool cm = cl > 0, cp = cl + 1 < M;
          int soff[MS];
          bool scol[MS];
#pragma unroll
          for (int q = 0; q < MS; ++q) {
            soff[q] = ssx[q] * M + ssy[q];
            scol[q] = q < nS && cl + ssy[q] >= 0 && cl + ssy[q] < M;
          }
          // the stencil of point (kk, cl) at element c from the centre column's values above
          // (cm_), at (cc_) and below (cd_) it.  The row-neighbour, column-neighbour and
          // sandwich parts are summed in independent chains (a point and its mirror round
          // alike), then added.
          auto point = [&](int kk, int c, C cm_, C cc_, C cd_) {
            const C ul = cm ? uin[c - 1] : zero;
            const C urr = cp ? uin[c + 1] : zero;
            const C kd = cmul(cadd(V[kk], b0), cc_);
            C kr = cmul(V[M + kk], cm_);
            C kc = cmul(bm, ul);
            kr = cfma(V[2 * M + kk], cd_, kr);
            kc = cfma(bp, urr, kc);
            C ks = zero;
#pragma unroll
            for (int q = 0; q < MS; ++q)
              if (q < nS && (!DIAG || !((sdiag >> q) & 1) || kk == cl)) {  // secular projector: k = l only
                const int xx = kk + ssx[q];
                const C v = (scol[q] && xx >= 0 && xx < M) ? uin[c + soff[q]] : zero;
                const C gxv = (has_sep && xx >= 0 && xx < M) ? gxi[xx] : zero;
                ks = cfma(V[(6 + q) * M + kk], cadd(cscale(v, sy[q]), cmul(gxv, gyp[q])), ks);
              }
            return cadd(cadd(kd, cadd(kr, kc)), ks);
          };
          // RK4 combine of the point at element c with state yj (stage sum and compensated
          // state update)
          auto combine = [&](int c, C kv, C& yj) {
            C outv;
            C& av = AS[c];
            if (stage == 1) {
              outv = caxpy(dt * (T)0.5, kv, yj);
              av = kv;
            } else if (stage == 4) {
              const C sm = cadd(av, kv);
              C& cv = CS[c];
              const C cw = cv;
              C d, t;
              d.x = dt * (T)(1.0 / 6.0) * sm.x - cw.x;
              d.y = dt * (T)(1.0 / 6.0) * sm.y - cw.y;
              t.x = yj.x + d.x;
              t.y = yj.y + d.y;
              C cn;
              cn.x = (t.x - yj.x) - d.x;
              cn.y = (t.y - yj.y) - d.y;
              cv = cn;
              yj = t;
              outv = t;
            } else {
              outv = caxpy(stage == 2 ? dt * (T)0.5 : dt, kv, yj);
              av = caxpy((T)2, kv, av);
            }
            uout[c] = outv;
          };
          // two rows per iteration, both stencils computed in one block (independent chains
          // the compiler can interleave); the second row's is computed also where the strip
          // has ended (its reads stay inside the shared-memory arrays) and then dropped
          C um = k0 > 0 ? uin[(k0 - 1) * M + cl] : zero;
          C ucn = uin[k0 * M + cl];
#pragma unroll
          for (int j = 0; j < RB; j += 2) {
            const int kk = k0 + j;
            if (kk < k1) {
              const int c = kk * M + cl;
              const C u1 = kk + 1 < M ? uin[c + M] : zero;
              const C u2 = kk + 2 < M ? uin[c + 2 * M] : zero;
              const C kvA = point(kk, c, um, ucn, u1);
              const C kvB = point(kk + 1, c + M, ucn, u1, u2);
              combine(c, kvA, yv[j]);
              if (kk + 1 < k1) combine(c + M, kvB, yv[j + 1]);
              um = u1;
              ucn = u2;
            }
          }
        }
        if (gown) {
          const bool isx = gq < M;
          const int g = isx ? gq : gq - M;
          const C* gs = isx ? gxi : gyi;
          const C lo = g > 0 ? gs[g - 1] : zero, hi = g + 1 < M ? gs[g + 1] : zero;
          C kv;
          if (isx) {
            kv = cmul(cadd(V[g], Cc), gs[g]);
            kv = cfma(V[M + g], lo, kv);
            kv = cfma(V[2 * M + g], hi, kv);
          } else {
            kv = cmul(cadd(V[3 * M + g], mCc), gs[g]);
            kv = cfma(V[4 * M + g], lo, kv);
            kv = cfma(V[5 * M + g], hi, kv);
          }
          C outv;
          if (stage == 1) {
            outv = caxpy(dt * (T)0.5, kv, gy_v);
            ga_v = kv;
          } else if (stage == 4) {
            const C sm = cadd(ga_v, kv);
            C d, t;
            d.x = dt * (T)(1.0 / 6.0) * sm.x - gc_v.x;
            d.y = dt * (T)(1.0 / 6.0) * sm.y - gc_v.y;
            t.x = gy_v.x + d.x;
            t.y = gy_v.y + d.y;
            gc_v.x = (t.x - gy_v.x) - d.x;
            gc_v.y = (t.y - gy_v.y) - d.y;
            gy_v = t;
            outv = t;
          } else {
            outv = caxpy(stage == 2 ? dt * (T)0.5 : dt, kv, gy_v);
            ga_v = caxpy((T)2, kv, ga_v);
          }
          uout[nr + gq] = outv;
        }
        // merged vectors of the next stage (its coefficients were evaluated two stages ago)
        build_mv((cbuf + 1) % 3, mbuf ^ 1);
        cbuf = (cbuf + 1) % 3;
        mbuf ^= 1;
        __syncthreads();
      }
    }
#pragma unroll
    for (int j = 0; j < RB; ++j) {
      const int kk = k0 + j;
      if (kk < k1) {
        y_g[gidx_r(kk)] = yv[j];
        comp_g[gidx_r(kk)] = CS[kk * M + cl];
      }
    }
    if (gown) {
      y_g[g_gi] = gy_v;
      comp_g[g_gi] = gc_v;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------
// Observables: one warp per evaluation group, lanes over (initial condition, entry) pairs.
// The value of a state element is y - comp (comp: the rounding residual of the last update).
// ---------------------------------------------------------------------------------------
template <typename C>
struct StateView {
  const C* y;
  const C* c;
  __device__ __forceinline__ C operator[](int64_t i) const {
    const C a = y[i], b = c[i];
    C r;
    r.x = a.x - b.x;
    r.y = a.y - b.y;
    return r;
  }
};

// The error word next to the results (in the slot before the first), so that the host reads both with
// one copy: two pageable copies were 16 of the 69 us of a one-step call and its observable.
__device__ __forceinline__ void out_error(const unsigned int* error, double2* out) {
  if (error) out[-1] = make_double2((double)*error, 0.0);
}

template <typename T>
__global__ void k_eval(const SysDesc* __restrict__ sys, const EvalGroup* __restrict__ groups,
                       const EvalEntry* __restrict__ entries, const void* ystate, const void* cstate, double2* out,
                       int n_groups, const unsigned int* error) {
  using C = typename C2T<T>::type;
  if (blockIdx.x == 0 && threadIdx.x == 0) out_error(error, out);
  const StateView<C> y{reinterpret_cast<const C*>(ystate), reinterpret_cast<const C*>(cstate)};
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= n_groups) return;
  const EvalGroup g = groups[warp];
  double re = 0.0, im = 0.0;
  const int total = g.n_sys * g.n_e;
  for (int i = lane; i < total; i += 32) {
    const int s = i / g.n_e;
    const int e = i - s * g.n_e;
    const SysDesc& sd = sys[g.sys_off + s];
    const EvalEntry en = entries[g.e_off + e];
    double vr = 0.0, vi = 0.0;
    if (sd.has_sep) {
      const C a = y[sd.off_gx + en.kx];
      const C b = y[sd.off_gy + en.ly];
      vr += (double)a.x * (double)b.x - (double)a.y * (double)b.y;
      vi += (double)a.x * (double)b.y + (double)a.y * (double)b.x;
    }
    if (sd.has_r) {
      const C r = sd.r_diag ? (en.kx == en.ly ? y[sd.off_r + en.kx] : cmk<C>(0.0, 0.0))
                            : y[sd.off_r + (int64_t)en.kx * sd.n_g + en.ly];
      vr += (double)r.x;
      vi += (double)r.y;
    }
    // w * f * v
    const double fr = sd.w_re * en.f_re - sd.w_im * en.f_im;
    const double fi = sd.w_re * en.f_im + sd.w_im * en.f_re;
    re += fr * vr - fi * vi;
    im += fr * vi + fi * vr;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    re += __shfl_down_sync(0xffffffffu, re, o);
    im += __shfl_down_sync(0xffffffffu, im, o);
  }
  if (lane == 0) out[warp] = make_double2(re, im);
}

// Observables for groups with few (initial condition, entry) pairs: one thread per group.
template <typename T>
__global__ void k_eval_small(const SysDesc* __restrict__ sys, const EvalGroup* __restrict__ groups,
                             const EvalEntry* __restrict__ entries, const void* ystate, const void* cstate, double2* out,
                             int n_groups, const unsigned int* error) {
  using C = typename C2T<T>::type;
  if (blockIdx.x == 0 && threadIdx.x == 0) out_error(error, out);
  const StateView<C> y{reinterpret_cast<const C*>(ystate), reinterpret_cast<const C*>(cstate)};
  const int gi = blockIdx.x * blockDim.x + threadIdx.x;
  if (gi >= n_groups) return;
  const EvalGroup g = groups[gi];
  double re = 0.0, im = 0.0;
  for (int s = 0; s < g.n_sys; ++s) {
    const SysDesc& sd = sys[g.sys_off + s];
    const double wr = sd.w_re, wim = sd.w_im;
    const int sep = sd.has_sep, hr = sd.has_r, ng = sd.n_g;
    const int64_t ox = sd.off_gx, oy = sd.off_gy, orr = sd.off_r;
    for (int e = 0; e < g.n_e; ++e) {
      const EvalEntry en = entries[g.e_off + e];
      double vr = 0.0, vi = 0.0;
      if (sep) {
        const C a = y[ox + en.kx];
        const C b = y[oy + en.ly];
        vr += (double)a.x * (double)b.x - (double)a.y * (double)b.y;
        vi += (double)a.x * (double)b.y + (double)a.y * (double)b.x;
      }
      if (hr) {
        const C r = sd.r_diag ? (en.kx == en.ly ? y[orr + en.kx] : cmk<C>(0.0, 0.0))
                              : y[orr + (int64_t)en.kx * ng + en.ly];
        vr += (double)r.x;
        vi += (double)r.y;
      }
      const double fr = wr * en.f_re - wim * en.f_im;
      const double fi = wr * en.f_im + wim * en.f_re;
      re += fr * vr - fi * vi;
      im += fr * vi + fi * vr;
    }
  }
  out[gi] = make_double2(re, im);
}

// Initial state: y[off] = value for a list of (offset, value) pairs (the rest is zeroed).
template <typename T>
__global__ void k_scatter(const InitEntry* __restrict__ ent, int n, void* ystate) {
  using C = typename C2T<T>::type;
  C* y = reinterpret_cast<C*>(ystate);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[ent[i].off] = cmk<C>(ent[i].re, ent[i].im);
}

// ---------------------------------------------------------------------------------------
// Fixed RK4 scratch for callers that cannot allocate device memory.
//
// bq_step_fixed_scratch() takes the two stage buffers and the RK4 accumulator from this
// file-scope array instead of from the state's pool.  Every GPU that loads the library
// holds it until the process exits.  Host code must not use the symbol's name as an
// address: fixed_scratch() looks the device address up once per device.
// ---------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_fixed_scratch[3 * BQ_FIXED_SCRATCH_BYTES];

cudaError_t fixed_scratch(void** ptr) {
  static std::mutex mu;
  static void* cache[256] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 256) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (!cache[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_fixed_scratch);
    if (e != cudaSuccess) return e;
    cache[dev] = p;
  }
  *ptr = cache[dev];
  return cudaSuccess;
}

// ---------------------------------------------------------------------------------------
// Host-side launchers.
// ---------------------------------------------------------------------------------------
template <typename T, int NM>
static cudaError_t launch_stage_t(const StageArgs& a, int n_work, int smem_bytes, cudaStream_t s) {
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(k_stage<T, NM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         BQ_MAX_DYN_SMEM);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  k_stage<T, NM><<<n_work, BQ_BLOCK, smem_bytes, s>>>(a);
  return cudaGetLastError();
}

template <typename T, int MX, int MY, int MS>
static cudaError_t launch_stage_m1_t(const StageArgs& a, const M1Sys* m1, int n_work, int smem_bytes, cudaStream_t s) {
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(k_stage_m1<T, MX, MY, MS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         BQ_MAX_DYN_SMEM);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  k_stage_m1<T, MX, MY, MS><<<n_work, BQ_BLOCK, smem_bytes, s>>>(a, m1);
  return cudaGetLastError();
}

cudaError_t launch_stage_m1(const StageArgs& a, const M1Sys* m1, int variant, int dtype, int n_work, int smem_bytes,
                            cudaStream_t s) {
  // variant 0: at most 2 terms per side; variant 1: at most BQ_M1_MAXT
  if (dtype == 0)
    return variant == 0 ? launch_stage_m1_t<double, 2, 2, 2>(a, m1, n_work, smem_bytes, s)
                        : launch_stage_m1_t<double, BQ_M1_MAXT, BQ_M1_MAXT, BQ_M1_MAXT>(a, m1, n_work, smem_bytes, s);
  return variant == 0 ? launch_stage_m1_t<float, 2, 2, 2>(a, m1, n_work, smem_bytes, s)
                      : launch_stage_m1_t<float, BQ_M1_MAXT, BQ_M1_MAXT, BQ_M1_MAXT>(a, m1, n_work, smem_bytes, s);
}

template <typename T, int BLK, int PPT>
static cudaError_t launch_solve_t(const SolveArgs& a, int smem_bytes, int cap_per_sm, cudaStream_t s, int* grid_out) {
  auto kern = a.has_diag ? k_solve_m1<T, BLK, PPT, 2, 2, 2, true> : k_solve_m1<T, BLK, PPT, 2, 2, 2, false>;
  {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, BQ_MAX_DYN_SMEM);
    if (e != cudaSuccess) return e;
  }
  int dev = 0, nsm = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, BLK, smem_bytes);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  if (cap_per_sm > 0) per_sm = std::min(per_sm, cap_per_sm);
  const int grid = std::min(a.n_sys, per_sm * nsm);
  *grid_out = grid;
  kern<<<grid, BLK, smem_bytes, s>>>(a);
  return cudaGetLastError();
}

template <typename T, int BLK, int RB>
static cudaError_t launch_solve_mg_t(const SolveArgs& a, int smem_bytes, int cap_per_sm, cudaStream_t s, int* grid_out) {
  auto kern = a.has_diag ? k_solve_mg<T, BLK, RB, BQ_M1_MAXT, BQ_M1_MAXT, 2, true>
                         : k_solve_mg<T, BLK, RB, BQ_M1_MAXT, BQ_M1_MAXT, 2, false>;
  {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, BQ_MAX_DYN_SMEM);
    if (e != cudaSuccess) return e;
  }
  int dev = 0, nsm = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, BLK, smem_bytes);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  if (cap_per_sm > 0) per_sm = std::min(per_sm, cap_per_sm);
  const int grid = std::min(a.n_sys, per_sm * nsm);
  *grid_out = grid;
  kern<<<grid, BLK, smem_bytes, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_solve_mg(const SolveArgs& a, int dtype, int smem_bytes, int cap_per_sm, cudaStream_t s,
                            int* grid_out) {
  // 256 threads; column strips of an even number of rows, at most 8 (M <= 42)
  return dtype == 0 ? launch_solve_mg_t<double, 256, 8>(a, smem_bytes, cap_per_sm, s, grid_out)
                    : launch_solve_mg_t<float, 256, 8>(a, smem_bytes, cap_per_sm, s, grid_out);
}

cudaError_t launch_solve_m1(const SolveArgs& a, int dtype, int capacity_class, int smem_bytes, int cap_per_sm,
                            cudaStream_t s, int* grid_out) {
  // capacity: FP32 256 threads x 7 points = 1792, FP64 448 threads x 4 points = 1792 points per system
  if (capacity_class != 0) return cudaErrorInvalidValue;
  return dtype == 0 ? launch_solve_t<double, 448, 4>(a, smem_bytes, cap_per_sm, s, grid_out)
                    : launch_solve_t<float, 256, 7>(a, smem_bytes, cap_per_sm, s, grid_out);
}

template <typename T, int NM>
static cudaError_t launch_adj_t(const AdjArgs& a, int n_work, int smem_bytes, int n_sys, int max_s, cudaStream_t s) {
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(k_adj_stage<T, NM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         BQ_MAX_DYN_SMEM);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  if (max_s > 0) {
    const int tiles = (a.ng_max + BQ_SRC_TILE - 1) / BQ_SRC_TILE;
    k_adj_src<T, NM><<<dim3(n_sys, max_s, 2 * tiles), BQ_SRC_THREADS, 0, s>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  k_adj_stage<T, NM><<<n_work, BQ_BLOCK, smem_bytes, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_adjoint(const AdjArgs& a, int dtype, int nm, int n_work, int smem_bytes, int n_sys, int max_s,
                           cudaStream_t s) {
  if (dtype == 0) {
    switch (nm) {
      case 1: return launch_adj_t<double, 1>(a, n_work, smem_bytes, n_sys, max_s, s);
      case 2: return launch_adj_t<double, 2>(a, n_work, smem_bytes, n_sys, max_s, s);
      case 3: return launch_adj_t<double, 3>(a, n_work, smem_bytes, n_sys, max_s, s);
      case 4: return launch_adj_t<double, 4>(a, n_work, smem_bytes, n_sys, max_s, s);
    }
  } else {
    switch (nm) {
      case 1: return launch_adj_t<float, 1>(a, n_work, smem_bytes, n_sys, max_s, s);
      case 2: return launch_adj_t<float, 2>(a, n_work, smem_bytes, n_sys, max_s, s);
      case 3: return launch_adj_t<float, 3>(a, n_work, smem_bytes, n_sys, max_s, s);
      case 4: return launch_adj_t<float, 4>(a, n_work, smem_bytes, n_sys, max_s, s);
    }
  }
  return cudaErrorInvalidValue;
}

// Cooperative segment kernels: the kernel for (dtype, modes, direction), its dynamic shared
// memory limit set once (static + dynamic within the per-block maximum).
template <typename T, int NM>
static const void* coop_kernel(bool bwd) {
  return bwd ? (const void*)k_coop_bwd<T, NM> : (const void*)k_coop_fwd<T, NM>;
}

static const void* coop_func(int dtype, int nm, bool bwd) {
  if (dtype == 0) {
    switch (nm) {
      case 1: return coop_kernel<double, 1>(bwd);
      case 2: return coop_kernel<double, 2>(bwd);
      case 3: return coop_kernel<double, 3>(bwd);
      case 4: return coop_kernel<double, 4>(bwd);
    }
  } else {
    switch (nm) {
      case 1: return coop_kernel<float, 1>(bwd);
      case 2: return coop_kernel<float, 2>(bwd);
      case 3: return coop_kernel<float, 3>(bwd);
      case 4: return coop_kernel<float, 4>(bwd);
    }
  }
  return nullptr;
}

static cudaError_t coop_prepare(const void* f, int smem_bytes) {
  static std::mutex mu;
  static std::vector<const void*> done;
  std::lock_guard<std::mutex> lock(mu);
  for (const void* d : done)
    if (d == f) return cudaSuccess;
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, f);
  if (e != cudaSuccess) return e;
  int dev = 0, optin = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  const int lim = std::min<int>(BQ_MAX_DYN_SMEM, optin - (int)fa.sharedSizeBytes);
  if (smem_bytes > lim) return cudaErrorInvalidValue;
  e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  if (e != cudaSuccess) return e;
  done.push_back(f);
  return cudaSuccess;
}

cudaError_t coop_max_grid(int dtype, int nm, bool bwd, int smem_bytes, int* out) {
  const void* f = coop_func(dtype, nm, bwd);
  if (!f) return cudaErrorInvalidValue;
  cudaError_t e = coop_prepare(f, smem_bytes);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, coop = 0, per_sm = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, BQ_BLOCK, smem_bytes);
  if (e != cudaSuccess) return e;
  *out = coop ? per_sm * sms : 0;
  return cudaSuccess;
}

cudaError_t launch_coop(int dtype, int nm, bool bwd, CoopArgs P, int smem_bytes, int grid, cudaStream_t s) {
  const void* f = coop_func(dtype, nm, bwd);
  if (!f || grid < 1) return cudaErrorInvalidValue;
  cudaError_t e = coop_prepare(f, smem_bytes);
  if (e != cudaSuccess) return e;
  P.src_tiles = (P.adj.ng_max + BQ_SRC_TILE_COOP - 1) / BQ_SRC_TILE_COOP;
  void* args[] = {(void*)&P};
  return cudaLaunchCooperativeKernel(f, dim3(grid), dim3(BQ_BLOCK), args, (size_t)smem_bytes, s);
}

cudaError_t launch_adj_seed(const SysDesc* sys, const EvalGroup* groups, const EvalEntry* entries, const void* y,
                            void* lam, int n_groups, int dtype, cudaStream_t s) {
  if (n_groups <= 0) return cudaSuccess;
  const int blocks = (n_groups + 127) / 128;
  if (dtype == 0)
    k_adj_seed<double><<<blocks, 128, 0, s>>>(sys, groups, entries, y, lam, n_groups);
  else
    k_adj_seed<float><<<blocks, 128, 0, s>>>(sys, groups, entries, y, lam, n_groups);
  return cudaGetLastError();
}

// The pipelined stage kernel for (dtype, variant, stage): variant 0 = at most 2 terms per side,
// variant 1 = at most BQ_M1_MAXT.
template <typename T, int MXYS>
static auto pipe_kernel(int stage) {
  switch (stage) {
    case 1: return k_stage_pipe<T, MXYS, MXYS, MXYS, 1>;
    case 2: return k_stage_pipe<T, MXYS, MXYS, MXYS, 2>;
    case 3: return k_stage_pipe<T, MXYS, MXYS, MXYS, 3>;
    default: return k_stage_pipe<T, MXYS, MXYS, MXYS, 4>;
  }
}

template <typename T, int MXYS>
static cudaError_t pipe_attrs_t() {
  for (int stage = 1; stage <= 4; ++stage) {
    cudaError_t e = cudaFuncSetAttribute(pipe_kernel<T, MXYS>(stage), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         BQ_MAX_DYN_SMEM);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

static cudaError_t pipe_attrs() {
  static std::mutex mu;
  static bool done = false;
  std::lock_guard<std::mutex> lock(mu);
  if (done) return cudaSuccess;
  cudaError_t e;
  if ((e = pipe_attrs_t<double, 2>()) != cudaSuccess) return e;
  if ((e = pipe_attrs_t<double, BQ_M1_MAXT>()) != cudaSuccess) return e;
  if ((e = pipe_attrs_t<float, 2>()) != cudaSuccess) return e;
  if ((e = pipe_attrs_t<float, BQ_M1_MAXT>()) != cudaSuccess) return e;
  const void* steps[4] = {(const void*)k_steps_pipe<double, 2, 2, 2>,
                          (const void*)k_steps_pipe<double, BQ_M1_MAXT, BQ_M1_MAXT, BQ_M1_MAXT>,
                          (const void*)k_steps_pipe<float, 2, 2, 2>,
                          (const void*)k_steps_pipe<float, BQ_M1_MAXT, BQ_M1_MAXT, BQ_M1_MAXT>};
  for (const void* f : steps)
    if ((e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, BQ_MAX_DYN_SMEM)) != cudaSuccess)
      return e;
  done = true;
  return cudaSuccess;
}

cudaError_t launch_stage_pipe(const PipeArgs& a, int variant, int dtype, int stage, int grid, int smem_bytes,
                              cudaStream_t s) {
  cudaError_t ea = pipe_attrs();
  if (ea != cudaSuccess) return ea;
  if (stage < 1 || stage > 4) return cudaErrorInvalidValue;
  if (dtype == 0) {
    if (variant == 0) pipe_kernel<double, 2>(stage)<<<grid, BQ_PIPE_THREADS, smem_bytes, s>>>(a);
    else pipe_kernel<double, BQ_M1_MAXT>(stage)<<<grid, BQ_PIPE_THREADS, smem_bytes, s>>>(a);
  } else {
    if (variant == 0) pipe_kernel<float, 2>(stage)<<<grid, BQ_PIPE_THREADS, smem_bytes, s>>>(a);
    else pipe_kernel<float, BQ_M1_MAXT>(stage)<<<grid, BQ_PIPE_THREADS, smem_bytes, s>>>(a);
  }
  return cudaGetLastError();
}

// The multi-step kernel for (dtype, variant).
static const void* steps_pipe_func(int dtype, int variant) {
  if (dtype == 0)
    return variant == 0 ? (const void*)k_steps_pipe<double, 2, 2, 2>
                        : (const void*)k_steps_pipe<double, BQ_M1_MAXT, BQ_M1_MAXT, BQ_M1_MAXT>;
  return variant == 0 ? (const void*)k_steps_pipe<float, 2, 2, 2>
                      : (const void*)k_steps_pipe<float, BQ_M1_MAXT, BQ_M1_MAXT, BQ_M1_MAXT>;
}

cudaError_t launch_steps_pipe(const PipeArgs& a, void* ua, void* ub, int n_steps, int variant, int dtype, int grid,
                              int smem_bytes, cudaStream_t s) {
  cudaError_t ea = pipe_attrs();
  if (ea != cudaSuccess) return ea;
  if (n_steps < 1) return cudaSuccess;
  PipeArgs pa = a;
  void* args[] = {(void*)&pa, (void*)&ua, (void*)&ub, (void*)&n_steps};
  return cudaLaunchKernel(steps_pipe_func(dtype, variant), dim3(grid), dim3(BQ_PIPE_THREADS), args,
                          (size_t)smem_bytes, s);
}

cudaError_t steps_pipe_blocks_per_sm(int dtype, int variant, int smem_bytes, int* out) {
  cudaError_t ea = pipe_attrs();
  if (ea != cudaSuccess) return ea;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, steps_pipe_func(dtype, variant), BQ_PIPE_THREADS,
                                                       smem_bytes);
}

cudaError_t pipe_blocks_per_sm(int dtype, int variant, int stage, int smem_bytes, int* out) {
  cudaError_t ea = pipe_attrs();
  if (ea != cudaSuccess) return ea;
  if (stage < 1 || stage > 4) return cudaErrorInvalidValue;
  if (dtype == 0)
    return variant == 0
               ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, pipe_kernel<double, 2>(stage), BQ_PIPE_THREADS, smem_bytes)
               : cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, pipe_kernel<double, BQ_M1_MAXT>(stage), BQ_PIPE_THREADS,
                                                               smem_bytes);
  return variant == 0
             ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, pipe_kernel<float, 2>(stage), BQ_PIPE_THREADS, smem_bytes)
             : cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, pipe_kernel<float, BQ_M1_MAXT>(stage), BQ_PIPE_THREADS,
                                                             smem_bytes);
}

template <typename K>
static cudaError_t occupancy_with_smem(K kern, int threads, int smem_bytes, int* out) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, BQ_MAX_DYN_SMEM);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, kern, threads, smem_bytes);
}

cudaError_t solve_blocks_per_sm(int dtype, int merged, int smem_bytes, int* out) {
  if (merged)
    return dtype == 0 ? occupancy_with_smem(k_solve_mg<double, 256, 8, BQ_M1_MAXT, BQ_M1_MAXT, 2, false>, 256, smem_bytes, out)
                      : occupancy_with_smem(k_solve_mg<float, 256, 8, BQ_M1_MAXT, BQ_M1_MAXT, 2, false>, 256, smem_bytes, out);
  return dtype == 0 ? occupancy_with_smem(k_solve_m1<double, 448, 4, 2, 2, 2, false>, 448, smem_bytes, out)
                    : occupancy_with_smem(k_solve_m1<float, 256, 7, 2, 2, 2, false>, 256, smem_bytes, out);
}

cudaError_t launch_stage(const StageArgs& a, int dtype, int nm, int n_work, int smem_bytes, cudaStream_t s) {
  if (dtype == 0) {
    switch (nm) {
      case 1: return launch_stage_t<double, 1>(a, n_work, smem_bytes, s);
      case 2: return launch_stage_t<double, 2>(a, n_work, smem_bytes, s);
      case 3: return launch_stage_t<double, 3>(a, n_work, smem_bytes, s);
      case 4: return launch_stage_t<double, 4>(a, n_work, smem_bytes, s);
    }
  } else {
    switch (nm) {
      case 1: return launch_stage_t<float, 1>(a, n_work, smem_bytes, s);
      case 2: return launch_stage_t<float, 2>(a, n_work, smem_bytes, s);
      case 3: return launch_stage_t<float, 3>(a, n_work, smem_bytes, s);
      case 4: return launch_stage_t<float, 4>(a, n_work, smem_bytes, s);
    }
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_eval(const SysDesc* sys, const EvalGroup* groups, const EvalEntry* entries, const void* y,
                        const void* comp, double2* out, int n_groups, int dtype, int small, const unsigned int* error,
                        cudaStream_t s) {
  if (n_groups <= 0) return cudaSuccess;
  const int threads = 256;
  if (small) {
    const int blocks = (n_groups + threads - 1) / threads;
    if (dtype == 0)
      k_eval_small<double><<<blocks, threads, 0, s>>>(sys, groups, entries, y, comp, out, n_groups, error);
    else
      k_eval_small<float><<<blocks, threads, 0, s>>>(sys, groups, entries, y, comp, out, n_groups, error);
    return cudaGetLastError();
  }
  const int blocks = (n_groups * 32 + threads - 1) / threads;
  if (dtype == 0)
    k_eval<double><<<blocks, threads, 0, s>>>(sys, groups, entries, y, comp, out, n_groups, error);
  else
    k_eval<float><<<blocks, threads, 0, s>>>(sys, groups, entries, y, comp, out, n_groups, error);
  return cudaGetLastError();
}

// Tr(rho0_b A_b) of every problem from the per-system contributions the last pipelined stage
// left (Eq. 11: the sum over the problem's initial conditions), one thread per problem,
// summed in system order.
__global__ void k_obs_sum(const double2* __restrict__ obs, const EvalGroup* __restrict__ groups, int n_groups,
                          double2* __restrict__ out, const unsigned int* error) {
  if (blockIdx.x == 0 && threadIdx.x == 0) out_error(error, out);
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= n_groups) return;
  const EvalGroup gr = groups[g];
  double re = 0.0, im = 0.0;
  for (int i = 0; i < gr.n_sys; ++i) {
    const double2 v = obs[gr.sys_off + i];
    re += v.x;
    im += v.y;
  }
  out[g] = make_double2(re, im);
}

cudaError_t launch_obs_sum(const double2* obs, const EvalGroup* groups, int n_groups, double2* out, const unsigned int* error,
                           cudaStream_t s) {
  if (n_groups <= 0) return cudaSuccess;
  const int threads = 256;
  k_obs_sum<<<(n_groups + threads - 1) / threads, threads, 0, s>>>(obs, groups, n_groups, out, error);
  return cudaGetLastError();
}

cudaError_t launch_scatter(const InitEntry* ent, int n, void* y, int dtype, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int threads = 256;
  const int blocks = (n + threads - 1) / threads;
  if (dtype == 0)
    k_scatter<double><<<blocks, threads, 0, s>>>(ent, n, y);
  else
    k_scatter<float><<<blocks, threads, 0, s>>>(ent, n, y);
  return cudaGetLastError();
}

}  // namespace bq
