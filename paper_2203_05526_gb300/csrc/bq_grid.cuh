// Grid-resident kernels of multi-mode states: all steps of a call in one cooperative launch.
//
// A state of a few ten thousand points (two modes at N = 12: 21 000) is a chain of short
// dependent stages.  One launch per stage spent most of its 11 us on the launch, on reloading
// descriptors, on building coefficient tables and on integer work per term; the FP64 pipe was
// busy a third of the time.  Here every point stays with one lane for the whole call, its
// state, stage sum, compensation and stage input in shared memory; only the stage input is
// exchanged, through L2, with one grid barrier per stage.  Per point (k, l), k and l flat over the modes,
//   (dx_k + dy_l) u + sum_j a_j (xm_k u(k-d,l) - yp_l u(k,l+d)) - conj(a_j) (xp_k u(k+d,l) - ym_l u(k,l-d))
//   + sum_q sx_k sy_l (u(k+s,l+s) + G_x[k+s] G_y[l+s])
// with real static weights in tables of n_g entries (products over the modes, zero where the
// source leaves the grid) and one complex coefficient per pair of a Hermitian H's terms: two
// to three times fewer FP64 operations than term by term.  Hermitian states (see
// bq_resident.cuh for the layout) hold half the points.
// Measured (one GB300, FP64, per RK4 step): two modes at N = 12 45 -> 20 us, three modes at N = 6
// direct 183 -> 68, mapped with R(xy) (125 systems) 279 -> 66; the 131-parameter control gradient
// 201 -> 76.  What bounds a stage now: the barrier (1.3 us), one round trip to L2, and the FP64
// pipe (one warp instruction per 16 cycles and SM).
#pragma once

#include "bq_device.cuh"
#include "bq_grid.h"

namespace bq {

#define BQ_GRID_WAIT_CYCLES2 (4000000000LL)  // about 2 s at the maximum SM clock

template <typename C> __device__ __forceinline__ C ld_cg(const C* p);
template <> __device__ __forceinline__ float2 ld_cg<float2>(const float2* p) { return __ldcg(p); }
template <> __device__ __forceinline__ double2 ld_cg<double2>(const double2* p) { return __ldcg(p); }

// Grid barrier number `round` (1, 2, ...) of a launch: one counter, zero before the launch, that
// every CTA adds one to; one thread per CTA waits for round x CTAs arrivals.  Measured on 152
// CTAs: 1.3 us; a word per CTA polled by everybody (no atomics) takes 6.5 us, the polls of 152 x
// 152 words delaying the stores they wait for.  The wait is bounded; on timeout the error word is
// set and the caller returns.  The CTA's earlier writes are visible to the others after it.
__device__ __forceinline__ bool grid_sync(unsigned int* bar, unsigned int round, unsigned int* error) {
  __syncthreads();
  int bad = 0;
  if (threadIdx.x == 0) {
    __threadfence();
    unsigned int v;
    asm volatile("atom.release.gpu.global.add.u32 %0, [%1], 1;" : "=r"(v) : "l"(bar) : "memory");
    const unsigned int want = round * gridDim.x;  // (wraps with the counter: compared as a difference)
    const long long t0 = clock64();
    for (;;) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if ((int)(v - want) >= 0) break;
      if (clock64() - t0 > BQ_GRID_WAIT_CYCLES2) {
        atomicOr(error, 4u);
        bad = 1;
        break;
      }
    }
  }
  return __syncthreads_or(bad) == 0;
}

template <typename T>
struct GridTab {
  using C = typename C2T<T>::type;
  const C *dx, *dy;
  const T* w;
  int ng, np, ns;
  // b: the problem's tables
  __device__ __forceinline__ GridTab(const GridProb& p, const T* b) : ng(p.ng), np(p.np), ns(p.ns) {
    dx = reinterpret_cast<const C*>(b);
    dy = dx + ng;
    w = b + 4 * ng;
  }
  __device__ __forceinline__ const T* pair(int j, int q) const { return w + (4 * j + q) * ng; }  // xm xp ym yp
  __device__ __forceinline__ const T* sand(int j, int q) const { return w + (4 * np + 2 * j + q) * ng; }
  __device__ __forceinline__ const T* pairT(int j, int q) const { return w + (4 * np + 2 * ns + 4 * j + q) * ng; }
  __device__ __forceinline__ const T* sandT(int j, int q) const { return w + (8 * np + 2 * ns + 2 * j + q) * ng; }
  __device__ __forceinline__ const C* diagp(int t, int q) const {
    return reinterpret_cast<const C*>(w + (8 * np + 4 * ns) * ng) + (2 * t + q) * ng;
  }
};

// Conjugate where m is the sign bit, unchanged where it is zero.
__device__ __forceinline__ float2 conj_bit(float2 v, unsigned m) {
  v.y = __uint_as_float(__float_as_uint(v.y) ^ m);
  return v;
}
__device__ __forceinline__ double2 conj_bit(double2 v, unsigned m) {
  v.y = __hiloint2double(__double2hiint(v.y) ^ (int)m, __double2loint(v.y));
  return v;
}

// a p - conj(a) q added to k; a purely imaginary a (uniform over the CTA) takes two
// multiply-adds per component less.
template <typename C>
__device__ __forceinline__ C pair_sum(C a, C p, C q, C k) {
  const C s = cadd(p, q);
  if (a.x == 0) {
    k.x = fma(-a.y, s.y, k.x);
    k.y = fma(a.y, s.x, k.y);
  } else {
    C d;
    d.x = p.x - q.x;
    d.y = p.y - q.y;
    k.x = fma(a.x, d.x, fma(-a.y, s.y, k.x));
    k.y = fma(a.x, d.y, fma(a.y, s.x, k.y));
  }
  return k;
}

// g += u v, summed in FP64 (an FP32 product is rounded to FP32 first, as in the other kernels).
__device__ __forceinline__ void grad_add(double2& g, double2 u, double2 v) { g = cfma(u, v, g); }
__device__ __forceinline__ void grad_add(double2& g, float2 u, float2 v) {
  const float2 p = cmul(u, v);
  g.x += (double)p.x;
  g.y += (double)p.y;
}

// Envelopes of the problem's pairs for the eight steps from s0 on (32 stages, one per lane), into
// half (s0 / 8) & 1 of E[2][32][MAXP].
// (seg, if not null: the piecewise-constant segments of the eight steps, [2][8][MAXP])
template <typename T>
__device__ __forceinline__ void grid_envelope(const GridArgs& A, const GridProb& P, typename C2T<T>::type* E, long long s0,
                                              int* seg = nullptr) {
  using C = typename C2T<T>::type;
  const int lane = threadIdx.x & 31;
  const double tau = A.tau0 + (double)(A.step0 + s0 + (lane >> 2)) * A.dt;
  const int stage = (lane & 3) + 1;
  const double t = pipe_chan_time(1, tau, stage, A.dt, A.horizon, A.reverse);
  const double tm = pipe_chan_time(2, tau, stage, A.dt, A.horizon, A.reverse);
  float t32[2];
  t32[0] = (float)t;
  t32[1] = (float)(t - (double)t32[0]);
  for (int j = 0; j < P.np; ++j) {
    C a = cmk<C>(P.a_re[j], P.a_im[j]);
    if (P.ch[j] >= 0) {
      C e = pipe_chan_value<T>(P.chan[P.ch[j]], A.chpar, t, tm, t32);
      if (P.cj[j]) e.y = -e.y;
      a = cmul(a, e);
    }
    E[(((s0 >> 3) & 1) * 32 + lane) * BQ_GRID_MAXP + j] = a;
    if (seg && stage == 1) {
      int sg = -1;
      if (P.ch[j] >= 0 && P.cd[P.ch[j]].kind == 2) {
        const ChanDesc& cd = P.cd[P.ch[j]];
        const double* c = A.chpar + cd.par_off;
        const int n_seg = (cd.n_par - 2) / 2;
        const double x = floor((tm - c[0]) / c[1]);
        if (x >= 0.0 && x < (double)n_seg) sg = (int)x;
      }
      seg[(((s0 >> 3) & 1) * 8 + (lane >> 2)) * BQ_GRID_MAXP + j] = sg;
    }
  }
}

// Where a point's element and its neighbours sit in the exchange arrays.  General layout: k n_g +
// l.  Hermitian layout (herm): rows d of P = n_g | 1 columns, k = (l + d) mod P; the element
// (k', l') is at row (k' - l') mod P of column l', or the conjugate of the one at (l', k').
struct GridPos {
  int ng, P, D, k, l, d;
  bool herm;
  // index of (k + ds, l + dt) relative to the system's R block; conj: sign bit of the imaginary part
  __device__ __forceinline__ int at(int ds, int dt, unsigned& conj) const {
    conj = 0u;
    if (!herm) return (k + ds) * ng + l + dt;
    int r = d + ds - dt, c = l + dt;  // row (may leave [0, D]) and column
    int kk = k + ds;
    if (c < 0) c += P;
    if (c >= P) c -= P;
    if (kk < 0) kk += P;
    if (kk >= P) kk -= P;
    if (r < 0) r += P;
    if (r >= P) r -= P;
    if (r > D) {
      conj = 0x80000000u;
      return (P - r) * P + kk;
    }
    return r * P + c;
  }
};

// A point's program in shared memory, written once per launch: where its neighbours are in the
// exchange arrays (element offsets; the sign bit marks a value to conjugate), their weights and
// its diagonal coefficient.  With index arithmetic and table look-ups out of the stages, a piece
// takes about 150 instructions a stage instead of 940 (two modes), and a stage is a short chain:
// independent loads from L2, multiply-adds, one store.
// n: point slots of the CTA; strides of n keep a warp's accesses on consecutive words.
template <typename T>
struct GridSlots {
  using C = typename C2T<T>::type;
  GridPiece* pc;
  C *v0, *v1, *v2, *v3, *dg;  // state, sum, compensation, input (the adjoint: lam, lacc, b)
  C* E;
  T* w;
  int *off, *fl;  // fl: bit 0 = a point of the grid, bit 1 = on the diagonal of a Hermitian system
  int n;
  __device__ __forceinline__ GridSlots(unsigned char* sm, int pieces, int nw, int no) : n(32 * pieces) {
    pc = reinterpret_cast<GridPiece*>(sm);
    v0 = reinterpret_cast<C*>(pc + pieces);
    v1 = v0 + n; v2 = v1 + n; v3 = v2 + n; dg = v3 + n;
    E = dg + n;
    w = reinterpret_cast<T*>(E + 2 * 32 * BQ_GRID_MAXP);
    off = reinterpret_cast<int*>(w + (size_t)nw * n);
    fl = off + (size_t)no * n;
  }
};

template <typename C>
__device__ __forceinline__ C ld_at(const C* b, int o) {  // the value at a program offset
  return conj_bit(ld_cg(b + (o & 0x7fffffff)), (unsigned)o & 0x80000000u);
}

template <typename T, int NP, int NS>
__global__ void __launch_bounds__(BQ_GRID_THREADS, 1) k_grid_fwd(const GridArgs A) {
  using C = typename C2T<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ GridProb P;
  const GridCta cta = A.ctas[blockIdx.x];
  for (int i = threadIdx.x; i < (int)(sizeof(GridProb) / 4); i += BQ_GRID_THREADS)
    reinterpret_cast<int*>(&P)[i] = reinterpret_cast<const int*>(A.probs + cta.prob)[i];
  __syncthreads();
  const int ng = P.ng, np = P.np, ns = P.ns;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = BQ_GRID_THREADS / 32;
  const GridSlots<T> S(smem_raw, cta.n, 4 * np + ns, 4 * np + 3 * ns);
  const int n = S.n;
  C* const E = S.E;
  const C zero = cmk<C>(0.0, 0.0);
  for (int i = tid; i < cta.n * (int)(sizeof(GridPiece) / 4); i += BQ_GRID_THREADS)
    reinterpret_cast<int*>(S.pc)[i] = reinterpret_cast<const int*>(A.pieces + cta.p0)[i];
  __syncthreads();
  C* ua = reinterpret_cast<C*>(A.ua);
  C* ub = reinterpret_cast<C*>(A.ub);
  auto slot = [&](long long i, int stage) -> C* {
    if (A.rec) return reinterpret_cast<C*>(A.rec + ((size_t)i * 4 + stage - 1) * A.arr);
    return (stage & 1) ? ua : ub;
  };
  const int Pc = ng | 1;
  auto position = [&](const GridPiece& g) {
    GridPos p;
    p.ng = ng;
    p.P = Pc;
    p.D = Pc / 2;
    p.herm = g.kind == GRID_H;
    p.d = 0;
    const int i = g.start + lane;
    p.k = p.l = i;
    if (g.kind == GRID_H) {
      p.d = i / Pc;
      p.l = i - p.d * Pc;
      p.k = p.l + p.d;
      if (p.k >= Pc) p.k -= Pc;
    } else if (g.kind == GRID_R) {
      p.k = i / ng;
      p.l = i - p.k * ng;
    }
    return p;
  };
  // index of a lane's point in the exchange arrays
  auto xidx = [&](const GridPiece& g) {
    return (g.kind <= GRID_D ? g.off_r : g.kind == GRID_X ? g.off_gx : g.off_gy) + g.start + lane;
  };

  // ---- programs and state ---------------------------------------------------------------------
  const GridTab<T> W(P, reinterpret_cast<const T*>(A.tab) + P.tab);
  for (int q = warp; q < cta.n; q += nw) {
    const GridPiece g = S.pc[q];
    const GridPos p = position(g);
    const int pi = 32 * q + lane, self = xidx(g);
    const bool ok = lane < g.len && p.k < ng && p.l < ng;
    const int si = lane < g.len ? self : xidx(g) - lane;  // (an address that exists)
    for (int j = 0; j < 4 * np + 3 * ns; ++j) S.off[j * n + pi] = si;
    for (int j = 0; j < 4 * np + ns; ++j) S.w[j * n + pi] = (T)0;
    C yv = zero, cv = zero, dg = zero;
    if (ok) {
      const int i = g.kind == GRID_H ? g.off_r + p.k * ng + p.l : self;
      yv = reinterpret_cast<const C*>(A.y)[i];
      if (!A.comp_zero) cv = reinterpret_cast<const C*>(A.comp)[i];
      if (g.kind <= GRID_D) dg = cadd(W.dx[p.k], W.dy[p.l]);
      else if (g.kind == GRID_X) dg = cadd(W.dx[p.k], cmk<C>(g.c_re, g.c_im));
      else dg = cadd(W.dy[p.k], cmk<C>(-g.c_re, -g.c_im));
      auto put = [&](int j, T w, int o, unsigned conj) {
        if (w == (T)0) return;
        S.w[j * n + pi] = w;
        S.off[j * n + pi] = (int)((unsigned)o | conj);
      };
      for (int j = 0; j < np; ++j) {
        const int d = P.dlt[j];
        unsigned c = 0u;
        if (g.kind <= GRID_H) {  // sources k - d, k + d, l - d, l + d
          int o = p.at(-d, 0, c);
          put(4 * j, W.pair(j, 0)[p.k], g.off_r + o, c);
          o = p.at(d, 0, c);
          put(4 * j + 1, W.pair(j, 1)[p.k], g.off_r + o, c);
          o = p.at(0, -d, c);
          put(4 * j + 2, W.pair(j, 2)[p.l], g.off_r + o, c);
          o = p.at(0, d, c);
          put(4 * j + 3, W.pair(j, 3)[p.l], g.off_r + o, c);
        } else if (g.kind >= GRID_X) {
          const int x = g.kind == GRID_X ? 0 : 2;
          put(4 * j, W.pair(j, x)[p.k], self - d, 0u);
          put(4 * j + 1, W.pair(j, x + 1)[p.k], self + d, 0u);
        }
      }
      if (g.kind <= GRID_D)
        for (int s = 0; s < ns; ++s) {
          const int d = P.ss[s];
          T ww = W.sand(s, 0)[p.k] * W.sand(s, 1)[p.l];
          if (P.sst[s] && (p.k / P.sst[s]) % P.sM[s] != (p.l / P.sst[s]) % P.sM[s]) ww = (T)0;
          if (ww == (T)0) continue;
          unsigned c = 0u;
          const int o = g.kind == GRID_D ? p.k + d : p.at(d, d, c);
          put(4 * np + s, ww, g.off_r + o, c);
          S.off[(4 * np + ns + s) * n + pi] = g.off_gx + p.k + d;
          S.off[(4 * np + 2 * ns + s) * n + pi] =
              g.kind == GRID_H ? (int)((unsigned)(g.off_gx + p.l + d) | 0x80000000u) : g.off_gy + p.l + d;
        }
    }
    S.fl[pi] = (ok ? 1 : 0) | (g.kind == GRID_H && p.d == 0 ? 2 : 0);
    S.v0[pi] = S.v3[pi] = yv;
    S.v1[pi] = zero;
    S.v2[pi] = cv;
    S.dg[pi] = dg;
    if (lane < g.len) slot(0, 1)[self] = yv;
  }
  if (warp == nw - 1) grid_envelope<T>(A, P, E, 0);
  unsigned int epoch = 1;
  if (!grid_sync(A.bar, epoch, A.error)) return;

  const T hh = (T)A.dt, h2 = (T)(0.5 * A.dt);
  const double wd = A.dt / 6.0;
  const T w_hi = (T)wd, w_lo = (T)(wd - (double)w_hi);
#pragma unroll 1
  for (int step = 0; step < A.n_steps; ++step) {
#pragma unroll 1
    for (int stage = 1; stage <= 4; ++stage) {
      const C* in = slot(step, stage);
      const bool more = step + 1 < A.n_steps;
      C* out = stage < 4 ? slot(step, stage + 1) : more ? slot(step + 1, 1) : nullptr;
      const C* Es = E + (((step >> 3) & 1) * 32 + (step & 7) * 4 + stage - 1) * BQ_GRID_MAXP;
#pragma unroll 1
      for (int q = warp; q < cta.n; q += nw) {
        const int kind = S.pc[q].kind, len = S.pc[q].len;
        const int pi = 32 * q + lane;
        const T* w = S.w + pi;
        const int* off = S.off + pi;
        const C u = S.v3[pi];
        C k = cmul(S.dg[pi], u);
        if (kind <= GRID_H) {
          // every load first: they are independent and come from L2
          C nb[4 * NP];
#pragma unroll
          for (int j = 0; j < 4 * NP; ++j)
            if (j < 4 * np) nb[j] = ld_at(in, off[j * n]);
#pragma unroll
          for (int j = 0; j < NP; ++j) {
            if (j >= np) break;
            const T w0 = w[(4 * j) * n], w1 = w[(4 * j + 1) * n], w2 = w[(4 * j + 2) * n], w3 = w[(4 * j + 3) * n];
            C a, b;
            a.x = fma(w0, nb[4 * j].x, -w3 * nb[4 * j + 3].x);
            a.y = fma(w0, nb[4 * j].y, -w3 * nb[4 * j + 3].y);
            b.x = fma(w1, nb[4 * j + 1].x, -w2 * nb[4 * j + 2].x);
            b.y = fma(w1, nb[4 * j + 1].y, -w2 * nb[4 * j + 2].y);
            k = pair_sum(Es[j], a, b, k);
          }
        } else if (kind >= GRID_X) {
          C lo[NP], hi[NP];
#pragma unroll
          for (int j = 0; j < NP; ++j)
            if (j < np) {
              lo[j] = ld_at(in, off[(4 * j) * n]);
              hi[j] = ld_at(in, off[(4 * j + 1) * n]);
            }
#pragma unroll
          for (int j = 0; j < NP; ++j) {
            if (j >= np) break;
            k = pair_sum(conj_bit(Es[j], kind == GRID_X ? 0u : 0x80000000u), cscale(lo[j], w[(4 * j) * n]),
                         cscale(hi[j], w[(4 * j + 1) * n]), k);
          }
        }
        if (kind <= GRID_D) {
          C sv[NS], sx[NS], sy[NS];
          T sw[NS];
          unsigned any = 0u;
#pragma unroll
          for (int s = 0; s < NS; ++s) {
            if (s >= ns) break;
            sw[s] = w[(4 * np + s) * n];
            // (terms restricted to the diagonal of a mode are absent from most warps)
            if (__any_sync(0xffffffffu, sw[s] != (T)0)) {
              any |= 1u << s;
              sv[s] = ld_at(in, off[(4 * np + s) * n]);
              if (P.has_sep) {
                sx[s] = ld_at(in, off[(4 * np + ns + s) * n]);
                sy[s] = ld_at(in, off[(4 * np + 2 * ns + s) * n]);
              }
            }
          }
#pragma unroll
          for (int s = 0; s < NS; ++s) {
            if (s >= ns) break;
            if (any >> s & 1) k = caxpy(sw[s], P.has_sep ? cfma(sx[s], sy[s], sv[s]) : sv[s], k);
          }
        }
        const int fl = S.fl[pi];
        if (fl & 2) k.y = (T)0;  // the diagonal of a Hermitian system is real
        C nu;
        if (stage < 4) {
          nu = caxpy(stage == 3 ? hh : h2, k, S.v0[pi]);
          S.v1[pi] = stage == 1 ? k : caxpy((T)2, k, S.v1[pi]);
        } else {
          const C yv = S.v0[pi];
          const C s = cadd(S.v1[pi], k), cv = S.v2[pi];
          C d, e;
          if constexpr (sizeof(T) == 4) {
            d.x = fma(w_hi, s.x, fma(w_lo, s.x, -cv.x));
            d.y = fma(w_hi, s.y, fma(w_lo, s.y, -cv.y));
            two_sum(yv, d, nu, e);
            S.v2[pi] = cneg(e);
          } else {  // (w_lo is zero)
            d.x = fma(w_hi, s.x, -cv.x);
            d.y = fma(w_hi, s.y, -cv.y);
            nu.x = yv.x + d.x;
            nu.y = yv.y + d.y;
            e.x = (nu.x - yv.x) - d.x;
            e.y = (nu.y - yv.y) - d.y;
            S.v2[pi] = e;
          }
          S.v0[pi] = nu;
        }
        S.v3[pi] = nu;
        if (out && lane < len) out[xidx(S.pc[q])] = nu;
      }
      if (stage == 1 && (step & 7) == 4 && (step | 7) + 1 < A.n_steps && warp == nw - 1)
        grid_envelope<T>(A, P, E, (step | 7) + 1);
      if (stage < 4 || more) {
        if (!grid_sync(A.bar, ++epoch, A.error)) return;
      }
    }
  }
  for (int q = warp; q < cta.n; q += nw) {
    const GridPiece g = S.pc[q];
    const int pi = 32 * q + lane;
    if (!(S.fl[pi] & 1)) continue;
    C* y = reinterpret_cast<C*>(A.y);
    C* c = reinterpret_cast<C*>(A.comp);
    const C yv = S.v0[pi], cv = S.v2[pi];
    if (g.kind == GRID_H) {
      const GridPos p = position(g);
      if (p.d) {
        y[g.off_r + p.l * ng + p.k] = conj_bit(yv, 0x80000000u);
        c[g.off_r + p.l * ng + p.k] = conj_bit(cv, 0x80000000u);
      }
      y[g.off_r + p.k * ng + p.l] = yv;
      c[g.off_r + p.k * ng + p.l] = cv;
    } else {
      y[xidx(g)] = yv;
      c[xidx(g)] = cv;
      if (A.herm && P.herm && g.kind == GRID_X) {
        y[g.off_gy + g.start + lane] = conj_bit(yv, 0x80000000u);
        c[g.off_gy + g.start + lane] = conj_bit(cv, 0x80000000u);
      }
    }
  }
}

// The adjoint of n_steps recorded steps, last first (see k_adj_stage in bq_kernels.cu for the
// recursion): q = J^T b with the transposed weights at the same neighbours, b of the previous
// stage exchanged through L2, one barrier per stage.  The transposed separable source needs, at a
// point of G, sums over a row or column of b_R, which is complete once the stage's barrier has
// passed: a warp per G point sums it directly, in the same phase as the points of R (no
// reduction phase of its own).  Parameter sums stay in registers: per pair u P^T b and u Q^T b,
// reduced into the gradient slots when an envelope changes its value and at the end.
template <typename T, int NP, int NS>
__global__ void __launch_bounds__(BQ_GRID_THREADS, 1) k_grid_adj(const GridArgs A) {
  using C = typename C2T<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[BQ_GRID_THREADS / 32][4 * NP + BQ_GRID_MAXT + 2];
  __shared__ int segs[2 * 8 * BQ_GRID_MAXP];
  __shared__ GridProb P;
  const GridCta cta = A.ctas[blockIdx.x];
  for (int i = threadIdx.x; i < (int)(sizeof(GridProb) / 4); i += BQ_GRID_THREADS)
    reinterpret_cast<int*>(&P)[i] = reinterpret_cast<const int*>(A.probs + cta.prob)[i];
  __syncthreads();
  const int ng = P.ng, np = P.np, ns = P.ns, nt = P.nt;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = BQ_GRID_THREADS / 32;
  const GridSlots<T> S(smem_raw, cta.n, 4 * np + ns + 2 * nt, 4 * np + ns);
  const int n = S.n;
  C* const E = S.E;
  // weights of the sandwich terms over the flat index (the sums over rows and columns of b_R)
  T* swt = reinterpret_cast<T*>(S.fl + n);
  const C zero = cmk<C>(0.0, 0.0);
  for (int i = tid; i < cta.n * (int)(sizeof(GridPiece) / 4); i += BQ_GRID_THREADS)
    reinterpret_cast<int*>(S.pc)[i] = reinterpret_cast<const int*>(A.pieces + cta.p0)[i];
  const GridTab<T> W(P, reinterpret_cast<const T*>(A.tab) + P.tab);
  for (int i = tid; i < 2 * ns * ng; i += BQ_GRID_THREADS) swt[i] = W.sand(0, 0)[i];
  __syncthreads();
  C* ba = reinterpret_cast<C*>(A.ua);
  C* bb = reinterpret_cast<C*>(A.ub);
  auto xidx = [&](const GridPiece& g) {
    return (g.kind <= GRID_D ? g.off_r : g.kind == GRID_X ? g.off_gx : g.off_gy) + g.start + lane;
  };
  const T hh = (T)A.dt, w6 = hh * (T)(1.0 / 6.0), w3 = hh * (T)(1.0 / 3.0), h2 = hh * (T)0.5;
  for (int q = warp; q < cta.n; q += nw) {
    const GridPiece g = S.pc[q];
    const int pi = 32 * q + lane;
    const bool ok = lane < g.len;
    const int self = xidx(g), si = ok ? self : self - lane, i = g.start + lane;
    const int k = g.kind == GRID_R ? i / ng : i, l = g.kind == GRID_R ? i - k * ng : i;
    for (int j = 0; j < 4 * np + ns; ++j) {
      S.off[j * n + pi] = si;
      S.w[j * n + pi] = (T)0;
    }
    for (int t = 0; t < 2 * nt; ++t) S.w[(4 * np + ns + t) * n + pi] = (T)0;
    C v = zero, dg = zero;
    if (ok) {
      v = reinterpret_cast<const C*>(A.lam)[self];
      ba[self] = cscale(v, w6);
      if (g.kind <= GRID_D) dg = cadd(W.dx[k], W.dy[l]);
      else if (g.kind == GRID_X) dg = cadd(W.dx[k], cmk<C>(g.c_re, g.c_im));
      else dg = cadd(W.dy[k], cmk<C>(-g.c_re, -g.c_im));
      auto put = [&](int j, T w, int o) {
        if (w == (T)0) return;
        S.w[j * n + pi] = w;
        S.off[j * n + pi] = o;
      };
      // transposed sources: xmT at k + d, xpT at k - d, ymT at l + d, ypT at l - d
      for (int j = 0; j < np; ++j) {
        const int d = P.dlt[j];
        if (g.kind == GRID_R) {
          put(4 * j, W.pairT(j, 0)[k], self + d * ng);
          put(4 * j + 1, W.pairT(j, 1)[k], self - d * ng);
          put(4 * j + 2, W.pairT(j, 2)[l], self + d);
          put(4 * j + 3, W.pairT(j, 3)[l], self - d);
        } else if (g.kind >= GRID_X) {
          const int x = g.kind == GRID_X ? 0 : 2;
          put(4 * j, W.pairT(j, x)[k], self + d);
          put(4 * j + 1, W.pairT(j, x + 1)[k], self - d);
        }
      }
      if (g.kind <= GRID_D) {
        for (int s = 0; s < ns; ++s) {
          T ww = W.sandT(s, 0)[k] * W.sandT(s, 1)[l];
          // (a restricted term shifts x and y alike: its source is on the diagonal of its mode
          // exactly when the point is)
          if (P.sst[s] && (k / P.sst[s]) % P.sM[s] != (l / P.sst[s]) % P.sM[s]) ww = (T)0;
          put(4 * np + s, ww, self - P.ss[s] * (g.kind == GRID_D ? 1 : ng + 1));
        }
      }
      for (int t = 0; t < nt; ++t) {
        const C h = g.kind <= GRID_D ? cadd(W.diagp(t, 0)[k], W.diagp(t, 1)[l])
                                     : (g.kind == GRID_X ? W.diagp(t, 0)[k] : W.diagp(t, 1)[k]);
        S.w[(4 * np + ns + 2 * t) * n + pi] = h.x;
        S.w[(4 * np + ns + 2 * t + 1) * n + pi] = h.y;
      }
    }
    S.v0[pi] = S.v1[pi] = v;
    S.v3[pi] = cscale(v, w6);
    S.dg[pi] = dg;
  }
  // parameter sums of this thread
  double2 ga[NP], gb[NP], dcs = make_double2(0.0, 0.0);
  double gt[BQ_GRID_MAXT];
#pragma unroll
  for (int j = 0; j < NP; ++j) ga[j] = gb[j] = make_double2(0.0, 0.0);
#pragma unroll
  for (int t = 0; t < BQ_GRID_MAXT; ++t) gt[t] = 0.0;
  const long long last = A.n_steps - 1;
  if (warp == nw - 1) grid_envelope<T>(A, P, E, last & ~7LL, segs);
  unsigned int epoch = 1;
  if (!grid_sync(A.bar, epoch, A.error)) return;

  auto seg_of = [&](long long i, int j) { return segs[(((i >> 3) & 1) * 8 + (i & 7)) * BQ_GRID_MAXP + j]; };

#pragma unroll 1
  for (long long it = last; it >= 0; --it) {
#pragma unroll 1
    for (int stage = 4; stage >= 1; --stage) {
      const C* in = (stage & 1) ? bb : ba;
      C* out = (stage & 1) ? ba : bb;
      const C* U = reinterpret_cast<const C*>(A.rec + ((size_t)it * 4 + stage - 1) * A.arr);
      const C* Es = E + (((it >> 3) & 1) * 32 + (it & 7) * 4 + stage - 1) * BQ_GRID_MAXP;
#pragma unroll 1
      for (int q = warp; q < cta.n; q += nw) {
        const GridPiece& g = S.pc[q];
        const int kind = g.kind, len = g.len;
        const int pi = 32 * q + lane;
        const T* w = S.w + pi;
        const int* off = S.off + pi;
        const C b = S.v3[pi];
        const bool ok = lane < len;
        const C u = ok ? U[xidx(g)] : zero;
        C qv = cmul(S.dg[pi], b);
        if (kind == GRID_R) {
          C nb[4 * NP], sv[NS];
#pragma unroll
          for (int j = 0; j < 4 * NP; ++j)
            if (j < 4 * np) nb[j] = ld_cg(in + off[j * n]);
          unsigned any = 0u;
#pragma unroll
          for (int s = 0; s < NS; ++s) {
            if (s >= ns) break;
            if (__any_sync(0xffffffffu, w[(4 * np + s) * n] != (T)0)) {
              any |= 1u << s;
              sv[s] = ld_cg(in + off[(4 * np + s) * n]);
            }
          }
#pragma unroll
          for (int j = 0; j < NP; ++j) {
            if (j >= np) break;
            const T w0 = w[(4 * j) * n], w1 = w[(4 * j + 1) * n], w2 = w[(4 * j + 2) * n], w3_ = w[(4 * j + 3) * n];
            C a, c;
            a.x = fma(w0, nb[4 * j].x, -w3_ * nb[4 * j + 3].x);
            a.y = fma(w0, nb[4 * j].y, -w3_ * nb[4 * j + 3].y);
            c.x = fma(w1, nb[4 * j + 1].x, -w2 * nb[4 * j + 2].x);
            c.y = fma(w1, nb[4 * j + 1].y, -w2 * nb[4 * j + 2].y);
            qv = pair_sum(Es[j], a, c, qv);
            if (P.gpar[j] >= 0 || P.gpwc[j] >= 0) {
              grad_add(ga[j], u, a);
              grad_add(gb[j], u, c);
            }
          }
#pragma unroll
          for (int s = 0; s < NS; ++s) {
            if (s >= ns) break;
            if (any >> s & 1) qv = caxpy(w[(4 * np + s) * n], sv[s], qv);
          }
        } else if (kind == GRID_D) {
          for (int s = 0; s < ns; ++s) qv = caxpy(w[(4 * np + s) * n], ld_cg(in + off[(4 * np + s) * n]), qv);
        } else {
          // points of G, BQ_GRID_GLEN per piece, the whole warp on each: the transposed source's
          // sum over a row (G_x) or column (G_y) of b_R, then the point's own lane the rest
          const bool isx = kind == GRID_X;
          C mine = zero;
          for (int gi = 0; gi < len && P.has_r && ns; ++gi) {
            const int k = g.start + gi;
            C src = zero;
            for (int s = 0; s < ns; ++s) {
              const int kk = k - P.ss[s];  // row / column of b_R
              if (kk < 0 || kk >= ng) continue;
              const T wt = swt[(2 * s + (isx ? 0 : 1)) * ng + kk];
              if (wt == (T)0) continue;
              const T* wo = swt + (2 * s + (isx ? 1 : 0)) * ng;
              const C* go = U + (isx ? g.off_gy : g.off_gx) + P.ss[s];
              C v = zero;
              if (P.r_diag) {
                if (lane == 0 && wo[kk] != (T)0) v = cmul(ld_cg(in + g.off_r + kk), cscale(go[kk], wo[kk]));
              } else {
                const C* br = in + g.off_r + (isx ? kk * ng : kk);
                const int st = isx ? 1 : ng;
                const int mk = P.sst[s] ? (kk / P.sst[s]) % P.sM[s] : 0;
                for (int j = lane; j < ng; j += 32) {
                  const T wj = wo[j];
                  if (wj == (T)0 || (P.sst[s] && (j / P.sst[s]) % P.sM[s] != mk)) continue;
                  v = cfma(ld_cg(br + j * st), cscale(go[j], wj), v);
                }
              }
              src = caxpy(wt, v, src);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
              src.x += __shfl_xor_sync(0xffffffffu, src.x, o);
              src.y += __shfl_xor_sync(0xffffffffu, src.y, o);
            }
            if (lane == gi) mine = src;
          }
          qv = cadd(qv, mine);
          if (ok) {
#pragma unroll
            for (int j = 0; j < NP; ++j) {
              if (j >= np) break;
              const C lo = cscale(ld_cg(in + off[(4 * j) * n]), w[(4 * j) * n]);
              const C hi = cscale(ld_cg(in + off[(4 * j + 1) * n]), w[(4 * j + 1) * n]);
              qv = pair_sum(conj_bit(Es[j], isx ? 0u : 0x80000000u), lo, hi, qv);
              if (P.gpar[j] >= 0 || P.gpwc[j] >= 0) {
                // X: a lo - conj(a) hi;  Y: conj(a) lo - a hi = a (-hi) - conj(a) (-lo)
                const C pa = isx ? lo : cneg(hi), pb = isx ? hi : cneg(lo);
                grad_add(ga[j], u, pa);
                grad_add(gb[j], u, pb);
              }
            }
            const C z = cmul(u, b);
            const double sg = isx ? 1.0 : -1.0;
            dcs.x += sg * (double)z.x;
            dcs.y += sg * (double)z.y;
          }
        }
        if (nt) {  // Re sum u b dD/dtheta of the parameters on diagonal terms
          const C z = cmul(u, b);
          for (int t = 0; t < BQ_GRID_MAXT; ++t) {
            if (t >= nt) break;
            const T hx = w[(4 * np + ns + 2 * t) * n], hy = w[(4 * np + ns + 2 * t + 1) * n];
            gt[t] += (double)(z.x * hx - z.y * hy);
          }
        }
        if (ok) {
          const C lv = S.v0[pi];
          const C av = cadd(S.v1[pi], qv);  // (the step's sum starts as lam)
          S.v1[pi] = av;
          C bn;
          if (stage > 1) {
            bn = caxpy(stage == 4 ? hh : h2, qv, cscale(lv, stage == 2 ? w6 : w3));
          } else {
            S.v0[pi] = av;
            bn = cscale(av, w6);
          }
          S.v3[pi] = bn;
          out[xidx(g)] = bn;
        }
      }
      // the eight steps below this batch, in its first step
      if (stage == 4 && ((it & 7) == 7 || it == last) && it > 7 && warp == nw - 1)
        grid_envelope<T>(A, P, E, (it & ~7LL) - 8, segs);
      // ---- parameter sums: reduced when a factor changes before the next stage, and at the end --
      bool flush = it == 0 && stage == 1;
      for (int j = 0; j < np && !flush; ++j) {
        if ((P.gpar[j] < 0 && P.gpwc[j] < 0) || P.ch[j] < 0) continue;
        const int kind = P.cd[P.ch[j]].kind;
        if (kind == 0) continue;
        if (kind != 2) flush = true;
        else if (stage == 1) flush = seg_of(it, j) != seg_of(it - 1, j);
      }
      if (flush) {  // (uniform over the CTA)
        auto sum = [&](double v) {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
          return v;
        };
#pragma unroll
        for (int j = 0; j < NP; ++j) {
          if (j >= np) break;
          const double x0 = sum(ga[j].x), x1 = sum(ga[j].y), x2 = sum(gb[j].x), x3 = sum(gb[j].y);
          if (lane == 0) {
            red[warp][4 * j] = x0; red[warp][4 * j + 1] = x1; red[warp][4 * j + 2] = x2; red[warp][4 * j + 3] = x3;
          }
          ga[j] = gb[j] = make_double2(0.0, 0.0);
        }
#pragma unroll
        for (int t = 0; t < BQ_GRID_MAXT; ++t) {
          const double x = sum(gt[t]);
          if (lane == 0) red[warp][4 * NP + t] = x;
          gt[t] = 0.0;
        }
        {
          const double x = sum(dcs.x), y = sum(dcs.y);
          if (lane == 0) {
            red[warp][4 * NP + BQ_GRID_MAXT] = x;
            red[warp][4 * NP + BQ_GRID_MAXT + 1] = y;
          }
          dcs = make_double2(0.0, 0.0);
        }
        __syncthreads();
        auto col = [&](int i) {
          double v = 0.0;
          for (int w = 0; w < nw; ++w) v += red[w][i];
          return v;
        };
        if (tid < np && (P.gpar[tid] >= 0 || P.gpwc[tid] >= 0)) {
          const int j = tid;
          const double2 sa = make_double2(col(4 * j), col(4 * j + 1)), sb = make_double2(col(4 * j + 2), col(4 * j + 3));
          double2 e = make_double2(1.0, 0.0);
          if (P.ch[j] >= 0) {
            const double tau = A.tau0 + (double)(A.step0 + it) * A.dt;
            const ChanDesc& cd = P.cd[P.ch[j]];
            const double t = pipe_chan_time(cd.kind == 2 ? 2 : 1, tau, stage, A.dt, A.horizon, A.reverse);
            const float t32[2] = {0.f, 0.f};
            e = pipe_chan_value<double>(P.chan[P.ch[j]], A.chpar, t, t, t32);
            if (P.cj[j]) e.y = -e.y;
          }
          // d Re(da S_a - conj(da) S_b) for a coefficient derivative da
          auto dre = [&](double2 da) {
            return da.x * sa.x - da.y * sa.y - (da.x * sb.x + da.y * sb.y);
          };
          if (P.gpar[j] >= 0) atomicAdd(A.grad + P.gpar[j], dre(cmul(make_double2(P.cb_re[j], P.cb_im[j]), e)));
          if (P.gpwc[j] >= 0) {
            const int sg = seg_of(it, j);
            if (sg >= 0) {
              const double2 c = make_double2(P.a_re[j], P.a_im[j]);
              const double2 ic = P.cj[j] ? make_double2(c.y, -c.x) : make_double2(-c.y, c.x);  // -+ i c
              atomicAdd(A.grad + P.gpwc[j] + 2 * sg, dre(c));
              atomicAdd(A.grad + P.gpwc[j] + 2 * sg + 1, dre(ic));
            }
          }
        }
        if (tid >= 32 && tid < 32 + nt) atomicAdd(A.grad + P.tpar[tid - 32], col(4 * NP + tid - 32));
        __syncthreads();
        // the separation constant's dependence on the parameters (an adjoint CTA holds one system)
        if (P.has_sep) {
          const double x = col(4 * NP + BQ_GRID_MAXT), y = col(4 * NP + BQ_GRID_MAXT + 1);
          for (int i = tid; i < P.n_params; i += BQ_GRID_THREADS) {
            const double2 v = A.dc[S.pc[0].dc_off + i];
            if (v.x != 0.0 || v.y != 0.0) atomicAdd(A.grad + P.grad_off + i, v.x * x - v.y * y);
          }
        }
        __syncthreads();
      }
      if (!(it == 0 && stage == 1)) {
        if (!grid_sync(A.bar, ++epoch, A.error)) return;
      }
    }
  }
  for (int q = warp; q < cta.n; q += nw) {
    const GridPiece& g = S.pc[q];
    if (lane < g.len) reinterpret_cast<C*>(A.lam)[xidx(g)] = S.v0[32 * q + lane];
  }
}

template <typename T>
static const void* grid_func_t(int np, int ns, bool adj) {
#define BQ_GRID_PICK(NPX, NSX) (adj ? (const void*)k_grid_adj<T, NPX, NSX> : (const void*)k_grid_fwd<T, NPX, NSX>)
  if (np <= 2) return ns <= 2 ? BQ_GRID_PICK(2, 2) : BQ_GRID_PICK(2, 4);
  if (np <= 4) return BQ_GRID_PICK(4, 4);
  return np <= BQ_GRID_MAXP && !adj ? (const void*)k_grid_fwd<T, 8, 4> : nullptr;
#undef BQ_GRID_PICK
}

static cudaError_t launch_grid_any(const void* f, const GridArgs& a, int ctas, int smem_bytes, cudaStream_t s) {
  if (!f || ctas < 1) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, BQ_GRID_SMEM_MAX);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(a.bar, 0, sizeof(unsigned int), s);
  if (e != cudaSuccess) return e;
  GridArgs p = a;
  void* args[] = {(void*)&p};
  return cudaLaunchCooperativeKernel(f, dim3(ctas), dim3(BQ_GRID_THREADS), args, (size_t)smem_bytes, s);
}

}  // namespace bq
