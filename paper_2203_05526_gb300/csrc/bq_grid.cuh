// Grid-resident kernels of multi-mode states: all steps of a call in one cooperative launch.
//
// A state of a few ten thousand points (two modes at N = 12: 21 000) is a chain of short
// dependent stages.  One launch per stage spent most of its 11 us on the launch, on reloading
// descriptors, on building coefficient tables and on integer work per term; the FP64 pipe was
// busy a third of the time.  Here every point stays with one lane for the whole call, its
// state, stage sum, compensation and stage input in shared memory; only the stage input is
// exchanged, through L2, in numbered slots that the readers poll (below: slots_wait).  Per point
// (k, l), k and l flat over the modes,
//   (dx_k + dy_l) u + sum_j a_j (xm_k u(k-d,l) - yp_l u(k,l+d)) - conj(a_j) (xp_k u(k+d,l) - ym_l u(k,l-d))
//   + sum_q sx_k sy_l (u(k+s,l+s) + G_x[k+s] G_y[l+s])
// with real static weights in tables of n_g entries (products over the modes, zero where the
// source leaves the grid) and one complex coefficient per pair of a Hermitian H's terms: two
// to three times fewer FP64 operations than term by term.  Hermitian states (see
// bq_resident.cuh for the layout) hold half the points.
// Measured (one GB300, FP64, per RK4 step; one launch per stage / a grid barrier per stage / slots):
// two modes at N = 12 45 / 20 / 9.8 us, three modes at N = 6 direct 183 / 68 / 28, mapped with R(xy)
// (125 systems) 279 / 66 / 37, with R = 0 88 / - / 20; the 131-parameter control gradient 201 / 76 / 46; one oscillator at N =
// 40, which the resident kernel keeps on one SM in 36 us, 9.  What bounds a stage now: small states
// the chain store, L2, poll, arithmetic of one warp (about 2 us); large ones the FP64 pipe (one warp
// instruction per 16 cycles and SM: 65% busy).
#pragma once

#include "bq_device.cuh"
#include "bq_grid.h"

namespace bq {

#define BQ_GRID_WAIT_CYCLES2 (4000000000LL)  // about 2 s at the maximum SM clock

// A launch's first grid barrier: one counter, zero before the launch, that every CTA adds one to; one
// thread per CTA waits for all.  The wait is bounded; on timeout the error word is set and the caller
// returns.  The CTA's earlier writes are visible to the others after it.
__device__ __forceinline__ bool grid_sync(unsigned int* bar, unsigned int* error) {
  __syncthreads();
  int bad = 0;
  if (threadIdx.x == 0) {
    unsigned int v;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    const long long t0 = clock64();
    for (;;) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if (v >= gridDim.x) break;
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
  const C* d;  // hi parts of dx, dy, then their lo parts
  const T* w;
  int ng, np, ns;
  // b: the problem's tables
  __device__ __forceinline__ GridTab(const GridProb& p, const T* b) : ng(p.ng), np(p.np), ns(p.ns) {
    d = reinterpret_cast<const C*>(b);
    w = b + 8 * ng;
  }
  // a + b + c, rounded (almost) once: a and b may cancel to far below their size
  static __device__ __forceinline__ C sum3(C a, C b, C c) {
    C s, e;
    two_sum(a, b, s, e);
    return cadd(s, cadd(e, c));
  }
  // diagonal coefficient of (k, l) of R, and of point k of G_x (side 0) or G_y (side 1) with c = C or -C
  __device__ __forceinline__ C diag(int k, int l) const { return sum3(d[k], d[ng + l], cadd(d[2 * ng + k], d[3 * ng + l])); }
  __device__ __forceinline__ C diag(int side, int k, double c_re, double c_im) const {
    const C hi = cmk<C>(c_re, c_im);
    return sum3(d[side * ng + k], hi, cadd(d[(2 + side) * ng + k], cmk<C>(c_re - (double)hi.x, c_im - (double)hi.y)));
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

// x == 0 on the integer pipe.
__device__ __forceinline__ bool zero_bits(double x) { return (__double_as_longlong(x) << 1) == 0; }
__device__ __forceinline__ bool zero_bits(float x) { return (__float_as_uint(x) << 1) == 0; }

// a p - conj(a) q added to k; a purely imaginary a (uniform over the CTA) takes two
// multiply-adds per component less.
template <typename C>
__device__ __forceinline__ C pair_sum(C a, C p, C q, C k) {
  const C s = cadd(p, q);
  if (zero_bits(a.x)) {
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

// g += a b + c d, summed in FP64 (FP32 products are rounded to FP32 first, as in the other kernels).
__device__ __forceinline__ void grad_add(double& g, double a, double b, double c, double d) { g = fma(a, b, fma(c, d, g)); }
__device__ __forceinline__ void grad_add(double& g, float a, float b, float c, float d) { g += (double)fmaf(a, b, c * d); }
__device__ __forceinline__ void grad_add(double& g, double a, double b) { g = fma(a, b, g); }
__device__ __forceinline__ void grad_add(double& g, float a, float b) { g += (double)(a * b); }

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

// ---- the exchange of stage inputs ----------------------------------------------------------------
// A slot is a value together with the number of the stage it is for, in 16-byte words {value,
// number} (FP64: one word per component; FP32: the value fits in one), each written and read as a
// whole (b128 accesses are single-copy atomic).  A reader polls the slots it needs until they carry
// its stage's number: no fence, no barrier, no flag between the writer's store and the reader's
// load.  A grid barrier per stage took four dependent trips to L2 (fence, counter, poll, load),
// this takes one and a half, and warps without a stage's last neighbours wait alone.
// Word of slot i in a place.  FP64: 32 slots' real words, then their imaginary words, so that a
// warp's 16-byte accesses are consecutive (a slot's two words side by side took twice the sectors:
// two modes 11.1 -> 12.9 us per step) and the second word is an immediate offset away.
template <typename C> __device__ __forceinline__ int slot_of(int i) { return sizeof(C) == 16 ? (i >> 5 << 6) | (i & 31) : i; }
__device__ __forceinline__ void slot_put(uint4* p, double2 v, unsigned int no) {
  asm volatile(
      "{\n.reg .b128 a, b;\nmov.b128 a, {%1, %3};\nmov.b128 b, {%2, %3};\n"
      "st.relaxed.gpu.global.b128 [%0], a;\nst.relaxed.gpu.global.b128 [%0+512], b;\n}" ::"l"(p),
      "l"(__double_as_longlong(v.x)), "l"(__double_as_longlong(v.y)), "l"((unsigned long long)no)
      : "memory");
}
__device__ __forceinline__ void slot_put(uint4* p, float2 v, unsigned int no) {
  const unsigned long long w = (unsigned long long)__float_as_uint(v.y) << 32 | __float_as_uint(v.x);
  asm volatile("{\n.reg .b128 a;\nmov.b128 a, {%1, %2};\nst.relaxed.gpu.global.b128 [%0], a;\n}" ::"l"(p), "l"(w),
               "l"((unsigned long long)no)
               : "memory");
}
// Zero if the slot carries the number.
__device__ __forceinline__ unsigned int slot_get(const uint4* p, unsigned int no, double2& v) {
  unsigned long long x, y, n0, n1;
  asm volatile(
      "{\n.reg .b128 a, b;\nld.relaxed.gpu.global.b128 a, [%4];\nld.relaxed.gpu.global.b128 b, [%4+512];\n"
      "mov.b128 {%0, %1}, a;\nmov.b128 {%2, %3}, b;\n}"
      : "=l"(x), "=l"(n0), "=l"(y), "=l"(n1)
      : "l"(p)
      : "memory");
  v.x = __longlong_as_double((long long)x);
  v.y = __longlong_as_double((long long)y);
  return ((unsigned int)n0 ^ no) | ((unsigned int)n1 ^ no);
}
__device__ __forceinline__ unsigned int slot_get(const uint4* p, unsigned int no, float2& v) {
  unsigned long long w, n0;
  asm volatile("{\n.reg .b128 a;\nld.relaxed.gpu.global.b128 a, [%2];\nmov.b128 {%0, %1}, a;\n}"
               : "=l"(w), "=l"(n0)
               : "l"(p)
               : "memory");
  v.x = __uint_as_float((unsigned int)w);
  v.y = __uint_as_float((unsigned int)(w >> 32));
  return (unsigned int)n0 ^ no;
}

// off(j): word of value j's slot; on: bit j set where value j is wanted (the
// others come back zero).  The whole warp calls it and stays together in the loop: when lanes left it
// one by one the arithmetic behind it was issued for several parts of the warp in turn (the FP64 pipe
// 93% busy for 44% of useful lanes, three modes direct).  The wait is bounded: a thread that gives up
// sets the error word and *dead, does not wait again, and the launch ends without storing.
template <int N, typename C, typename F>
__device__ __forceinline__ void slots_wait(const uint4* base, F off, unsigned int on, unsigned int no, C (&v)[N],
                                           unsigned int* error, int* dead) {
#pragma unroll
  for (int j = 0; j < N; ++j) v[j] = cmk<C>(0.0, 0.0);
  for (unsigned int tries = 1;; ++tries) {
    unsigned int bad = 0u;
#pragma unroll
    for (int j = 0; j < N; ++j)
      if (on >> j & 1u) bad |= slot_get(base + (unsigned)off(j), no, v[j]);
    if (!__any_sync(0xffffffffu, bad)) break;
    if (!(tries & 1023u)) {  // (a try takes a trip to L2: 2^22 of them about 2 s)
      const bool stop = tries >> 22;
      if (stop && bad) atomicOr(error, 4u);
      if (__any_sync(0xffffffffu, stop || *(volatile int*)dead)) {
        *(volatile int*)dead = 1;
        break;
      }
    }
  }
}
// The same for program offsets with the conjugation in their sign bit.
template <int N, typename C, typename F>
__device__ __forceinline__ void slots_wait_conj(const uint4* base, F off, unsigned int on, unsigned int no, C (&v)[N],
                                                unsigned int* error, int* dead) {
  slots_wait<N>(base, [&](int j) { return off(j) & 0x7fffffff; }, on, no, v, error, dead);
#pragma unroll
  for (int j = 0; j < N; ++j)
    if (on >> j & 1u) v[j] = conj_bit(v[j], (unsigned)off(j) & 0x80000000u);
}

// Slots are used in turn: stage number `no` has place no % ring.  On entering a block of `block`
// steps (block h = 1, 2, ...) a CTA counts itself and waits until all have entered block h - 1; every
// read of block h - 2 is then over, and its places (and one) may be written again: ring = 8 block +
// 1.  The wait is almost always over before it begins.  bar[0] is the launch's first barrier; block h
// counts in bar[1 + h % 4] (CTAs are never more than two blocks apart, so a word's counts of
// different blocks do not mix; one counter for all blocks would let fast CTAs stand in for slow ones).
__device__ __forceinline__ bool block_sync(unsigned int* bar, unsigned int h, unsigned int* error, int* dead) {
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar + 1 + (h & 3u)) : "memory");
    const unsigned int b = h - 1, want = ((b + 3u) >> 2) * gridDim.x;  // (wraps with the counter: compared as a difference)
    const long long t0 = clock64();
    while (b > 0) {
      unsigned int v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar + 1 + (b & 3u)) : "memory");
      if ((int)(v - want) >= 0) break;
      if (clock64() - t0 > BQ_GRID_WAIT_CYCLES2) {
        atomicOr(error, 4u);
        *(volatile int*)dead = 1;
        break;
      }
    }
  }
  return __syncthreads_or(threadIdx.x == 0 && *(volatile int*)dead) == 0;
}

// NPS > 0 (GRID_ONE): at most NPS pairs and NSS sandwich terms, a piece per warp: its state and its
// neighbours' slots stay in registers and every value comes in one batch of loads without a branch
// (a value that a point lacks is its own slot with a zero weight).  Else the
// program is read from shared memory and the pairs go in batches of two or, with 256 threads (no
// more than eight pieces a CTA, 255 registers), four.
template <typename T, int NPS, int NSS, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) k_grid_fwd(const GridArgs A) {
  using C = typename C2T<T>::type;
  constexpr bool SMALL = NPS > 0;
  constexpr int NV = SMALL ? 4 * NPS + 3 * NSS : 1;  // values of a point
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ GridProb P;
  __shared__ int dead;
  const GridCta cta = A.ctas[blockIdx.x];
  for (int i = threadIdx.x; i < (int)(sizeof(GridProb) / 4); i += THREADS)
    reinterpret_cast<int*>(&P)[i] = reinterpret_cast<const int*>(A.probs + cta.prob)[i];
  if (threadIdx.x == 0) dead = 0;
  __syncthreads();
  const int ng = P.ng, np = P.np, ns = P.ns;
  // pairs with a static imaginary coefficient i b: b is part of the weights
  unsigned int fold = 0u;
  for (int j = 0; j < np; ++j)
    if (P.ch[j] < 0 && P.a_re[j] == 0.0) fold |= 1u << j;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = THREADS / 32;
  const GridSlots<T> S(smem_raw, cta.n, 4 * np + ns, 4 * np + 3 * ns);
  const int n = S.n;
  C* const E = S.E;
  const C zero = cmk<C>(0.0, 0.0);
  for (int i = tid; i < cta.n * (int)(sizeof(GridPiece) / 4); i += THREADS)
    reinterpret_cast<int*>(S.pc)[i] = reinterpret_cast<const int*>(A.pieces + cta.p0)[i];
  __syncthreads();
  uint4* const ring = reinterpret_cast<uint4*>(A.ring);
  const size_t place = A.place;
  const int places = (int)min((long long)A.ring_places, 4LL * A.n_steps + 1);  // that this launch uses
  auto recorded = [&](long long i, int stage) { return reinterpret_cast<C*>(A.rec + ((size_t)i * 4 + stage - 1) * A.arr); };
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
    for (int j = 0; j < 4 * np + 3 * ns; ++j) S.off[j * n + pi] = slot_of<C>(si);
    for (int j = 0; j < 4 * np + ns; ++j) S.w[j * n + pi] = (T)0;
    C yv = zero, cv = zero, dg = zero;
    if (ok) {
      const int i = g.kind == GRID_H ? g.off_r + p.k * ng + p.l : self;
      yv = reinterpret_cast<const C*>(A.y)[i];
      if (!A.comp_zero) cv = reinterpret_cast<const C*>(A.comp)[i];
      if (g.kind <= GRID_D) dg = W.diag(p.k, p.l);
      else if (g.kind == GRID_X) dg = W.diag(0, p.k, g.c_re, g.c_im);
      else dg = W.diag(1, p.k, -g.c_re, -g.c_im);
      auto put = [&](int j, T w, int o, unsigned conj) {
        if (w == (T)0) return;
        S.w[j * n + pi] = w;
        S.off[j * n + pi] = (int)((unsigned)slot_of<C>(o) | conj);
      };
      for (int j = 0; j < np; ++j) {
        const int d = P.dlt[j];
        const T f = !(fold >> j & 1u) ? (T)1 : (T)(g.kind == GRID_Y ? -P.a_im[j] : P.a_im[j]);
        unsigned c = 0u;
        if (g.kind <= GRID_H) {  // sources k - d, k + d, l - d, l + d
          int o = p.at(-d, 0, c);
          put(4 * j, f * W.pair(j, 0)[p.k], g.off_r + o, c);
          o = p.at(d, 0, c);
          put(4 * j + 1, f * W.pair(j, 1)[p.k], g.off_r + o, c);
          o = p.at(0, -d, c);
          put(4 * j + 2, f * W.pair(j, 2)[p.l], g.off_r + o, c);
          o = p.at(0, d, c);
          put(4 * j + 3, f * W.pair(j, 3)[p.l], g.off_r + o, c);
        } else if (g.kind >= GRID_X) {
          const int x = g.kind == GRID_X ? 0 : 2;
          put(4 * j, f * W.pair(j, x)[p.k], self - d, 0u);
          put(4 * j + 1, f * W.pair(j, x + 1)[p.k], self + d, 0u);
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
          S.off[(4 * np + ns + s) * n + pi] = slot_of<C>(g.off_gx + p.k + d);
          S.off[(4 * np + 2 * ns + s) * n + pi] =
              g.kind == GRID_H ? (int)((unsigned)slot_of<C>(g.off_gx + p.l + d) | 0x80000000u) : slot_of<C>(g.off_gy + p.l + d);
        }
    }
    S.fl[pi] = (ok ? 1 : 0) | (g.kind == GRID_H && p.d == 0 ? 2 : 0);
    S.v0[pi] = S.v3[pi] = yv;
    S.v1[pi] = zero;
    S.v2[pi] = cv;
    S.dg[pi] = dg;
    if (g.kind <= GRID_D) {  // (terms restricted to the diagonal of a mode are absent from most warps)
      unsigned int any = 0u;
      for (int s = 0; s < ns; ++s)
        if (__any_sync(0xffffffffu, S.w[(4 * np + s) * n + pi] != (T)0)) any |= (P.has_sep ? 7u : 1u) << (3 * s);
      if (lane == 0) S.pc[q].pad = (int)any;
    }
    if (lane < g.len) {
      for (int r = 0; r < places; ++r)
        if (r != 1) slot_put(ring + r * place + slot_of<C>(self), zero, 0u);
      slot_put(ring + place + slot_of<C>(self), yv, 1u);
      if (A.rec) recorded(0, 1)[self] = yv;
    }
  }
  if (warp == nw - 1) grid_envelope<T>(A, P, E, 0);
  unsigned int block = 0;
  if (!grid_sync(A.bar, A.error)) return;

  const T hh = (T)A.dt, h2 = (T)(0.5 * A.dt);
  const double wd = A.dt / 6.0;
  const T w_hi = (T)wd, w_lo = (T)(wd - (double)w_hi);
  unsigned int no = 1;       // number and place of the stage's input
  const uint4* in = ring + place;
  int turn = 1;
  // the state after a step: y + (sum + k) dt / 6 with its rounding error carried along
  auto update = [&](C sum, C k, C yv, C& cv) {
    const C s = cadd(sum, k);
    C d, e, nu;
    if constexpr (sizeof(T) == 4) {
      d.x = fma(w_hi, s.x, fma(w_lo, s.x, -cv.x));
      d.y = fma(w_hi, s.y, fma(w_lo, s.y, -cv.y));
      two_sum(yv, d, nu, e);
      cv = cneg(e);
    } else {  // (w_lo is zero)
      d.x = fma(w_hi, s.x, -cv.x);
      d.y = fma(w_hi, s.y, -cv.y);
      if (A.single_mode) {
        sum_ordered(yv, d, nu, e);
        cv = cneg(e);
      } else {  // Fast2Sum, as the tiled kernel's: exact unless the increment is larger than the element
        nu.x = yv.x + d.x;
        nu.y = yv.y + d.y;
        cv.x = (nu.x - yv.x) - d.x;
        cv.y = (nu.y - yv.y) - d.y;
      }
    }
    return nu;
  };
  // a pair's contribution to k: values n0..n3 with weights w0..w3, coefficient a
  auto pair_term = [&](bool folded, C a, T w0, T w1, T w2, T w3, C n0, C n1, C n2, C n3, C& k) {
    if (folded) {  // k += i (w0 n0 + w1 n1 - w2 n2 - w3 n3)
      k.x = fma(w3, n3.y, fma(w2, n2.y, fma(-w1, n1.y, fma(-w0, n0.y, k.x))));
      k.y = fma(-w3, n3.x, fma(-w2, n2.x, fma(w1, n1.x, fma(w0, n0.x, k.y))));
      return;
    }
    C p;
    p.x = fma(w0, n0.x, -w3 * n3.x);
    p.y = fma(w0, n0.y, -w3 * n3.y);
    if (zero_bits(a.x)) {  // a = i b: the sum in one chain
      p.x = fma(w1, n1.x, fma(-w2, n2.x, p.x));
      p.y = fma(w1, n1.y, fma(-w2, n2.y, p.y));
      k.x = fma(-a.y, p.y, k.x);
      k.y = fma(a.y, p.x, k.y);
    } else {
      C b;
      b.x = fma(w1, n1.x, -w2 * n2.x);
      b.y = fma(w1, n1.y, -w2 * n2.y);
      k = pair_sum(a, p, b, k);
    }
  };
  // SMALL: a warp's one piece, its neighbours' slots, state, sum and compensation in registers
  int of[NV];
  unsigned int cj = 0u, sany = 0u;  // values to conjugate; sandwich terms present in the warp
  C y1 = zero, s1 = zero, c1 = zero, u1 = zero, dg1 = zero;
  int kind1 = 0, xi1 = -1, xs1 = 0;
  bool real1 = false;
  if (SMALL && warp < cta.n) {
    const GridPiece& g = S.pc[warp];
    const int pi = 32 * warp + lane, self = lane < g.len ? xidx(g) : xidx(g) - lane;
    kind1 = g.kind;
    if (lane < g.len) xi1 = self;
    xs1 = slot_of<C>(self);
    sany = (unsigned int)g.pad;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      // values 0 .. 4 NPS - 1: pairs (points of G have two of each four), then sandwich terms
      const int t = i - 4 * NPS, j = i < 4 * NPS ? i : 4 * np + t % 3 * ns + t / 3;
      const bool want = i < 4 * NPS ? i < 4 * np && kind1 != GRID_D && (kind1 <= GRID_H || (i & 3) < 2) : sany >> t & 1u;
      const int o = want ? S.off[j * n + pi] : slot_of<C>(self);
      of[i] = o & 0x7fffffff;
      cj |= ((unsigned)o >> 31) << i;
    }
    y1 = u1 = S.v0[pi];
    c1 = S.v2[pi];
    dg1 = S.dg[pi];
    real1 = S.fl[pi] & 2;
  }
#pragma unroll 1
  for (int step = 0; step < A.n_steps; ++step) {
    if (step > 0 && (step & (A.block - 1)) == 0) {
      if (!block_sync(A.bar, ++block, A.error, &dead)) return;
    }
    // (the next eight steps' envelopes: behind a block boundary, ahead of the one before their use)
    if ((step & 7) == 4 && (step | 7) + 1 < A.n_steps && warp == nw - 1) grid_envelope<T>(A, P, E, (step | 7) + 1);
#pragma unroll 1
    for (int stage = 1; stage <= 4; ++stage) {
      const bool send = stage < 4 || step + 1 < A.n_steps;
      turn = turn + 1 == A.ring_places ? 0 : turn + 1;
      uint4* out = ring + turn * place;
      const C* Es = E + (((step >> 3) & 1) * 32 + (step & 7) * 4 + stage - 1) * BQ_GRID_MAXP;
      if constexpr (SMALL) {
        if (warp < cta.n) {
          const T* w = S.w + 32 * warp + lane;
          C v[NV];
          slots_wait<NV>(in, [&](int i) { return of[i]; }, 0xffffffffu, no, v, A.error, &dead);
          if (kind1 == GRID_H) {
#pragma unroll
            for (int i = 0; i < NV; ++i) v[i] = conj_bit(v[i], cj << (31 - i) & 0x80000000u);
          }
          C k = cmul(dg1, u1);
          const unsigned int yc = kind1 == GRID_Y ? 0x80000000u : 0u;
#pragma unroll
          for (int j = 0; j < NPS; ++j)
            if (j < np && kind1 != GRID_D)
              pair_term(fold >> j & 1u, conj_bit(Es[j], yc), w[(4 * j) * n], w[(4 * j + 1) * n], w[(4 * j + 2) * n],
                        w[(4 * j + 3) * n], v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3], k);
#pragma unroll
          for (int s = 0; s < NSS; ++s)
            if (sany >> (3 * s) & 1u) {
              const int i = 4 * NPS + 3 * s;
              k = caxpy(w[(4 * np + s) * n], sany >> (3 * s + 1) & 1u ? cfma(v[i + 1], v[i + 2], v[i]) : v[i], k);
            }
          if (real1) k.y = (T)0;  // the diagonal of a Hermitian system is real
          if (stage < 4) {
            u1 = caxpy(stage == 3 ? hh : h2, k, y1);
            s1 = stage == 1 ? k : caxpy((T)2, k, s1);
          } else {
            y1 = u1 = update(s1, k, y1, c1);
          }
          if (send && xi1 >= 0) {
            slot_put(out + xs1, u1, no + 1);
            if (A.rec) (stage < 4 ? recorded(step, stage + 1) : recorded(step + 1, 1))[xi1] = u1;
          }
        }
      } else {
#pragma unroll 1
      for (int q = warp; q < cta.n; q += nw) {
        const int kind = S.pc[q].kind, len = S.pc[q].len;
        const unsigned int any = (unsigned int)S.pc[q].pad;
        const int pi = 32 * q + lane;
        const T* w = S.w + pi;
        const int* off = S.off + pi;
        const C u = S.v3[pi];
        C k = cmul(S.dg[pi], u);
        // pair j of R with its four neighbours, and a sandwich term with its three
        auto pair = [&](int j, C n0, C n1, C n2, C n3) {
          pair_term(fold >> j & 1u, Es[j], w[(4 * j) * n], w[(4 * j + 1) * n], w[(4 * j + 2) * n], w[(4 * j + 3) * n], n0, n1,
                    n2, n3, k);
        };
        auto sand = [&](int s, C v, C x, C y) {
          k = caxpy(w[(4 * np + s) * n], P.has_sep ? cfma(x, y, v) : v, k);
        };
        auto soff = [&](int i) { return off[(4 * np + (i % 3) * ns + i / 3) * n]; };  // value i of the sandwich terms
        if (kind >= GRID_X) {
#pragma unroll 1
          for (int j0 = 0; j0 < np; j0 += 4) {
            const int m = min(4, np - j0);
            C v[8];
            slots_wait_conj<8>(in, [&](int i) { return off[(4 * (j0 + i / 2) + (i & 1)) * n]; }, (1u << (2 * m)) - 1u, no, v,
                          A.error, &dead);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if (i >= m) break;
              const int j = j0 + i;
              const T w0 = w[(4 * j) * n], w1 = w[(4 * j + 1) * n];
              if (fold >> j & 1u) {
                k.x = fma(-w1, v[2 * i + 1].y, fma(-w0, v[2 * i].y, k.x));
                k.y = fma(w1, v[2 * i + 1].x, fma(w0, v[2 * i].x, k.y));
              } else {
                k = pair_sum(conj_bit(Es[j], kind == GRID_X ? 0u : 0x80000000u), cscale(v[2 * i], w0),
                             cscale(v[2 * i + 1], w1), k);
              }
            }
          }
        } else {
          constexpr int PB = THREADS == 256 ? 4 : 2;
          if (kind <= GRID_H) {
#pragma unroll 1
            for (int j0 = 0; j0 < np; j0 += PB) {
              const int m = min(PB, np - j0);
              C v[4 * PB];
              slots_wait_conj<4 * PB>(in, [&](int i) { return off[(4 * j0 + i) * n]; }, (1u << (4 * m)) - 1u, no, v, A.error, &dead);
#pragma unroll
              for (int i = 0; i < PB; ++i)
                if (i < m) pair(j0 + i, v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            }
          }
#pragma unroll 1
          for (int s0 = 0; s0 < ns; s0 += 2) {
            const unsigned int on = any >> (3 * s0) & 63u;
            if (!on) continue;
            C v[6];
            slots_wait_conj<6>(in, [&](int i) { return soff(3 * s0 + i); }, on, no, v, A.error, &dead);
#pragma unroll
            for (int s = 0; s < 2; ++s)
              if (on >> (3 * s) & 1u) sand(s0 + s, v[3 * s], v[3 * s + 1], v[3 * s + 2]);
          }
        }
        if (S.fl[pi] & 2) k.y = (T)0;  // the diagonal of a Hermitian system is real
        C nu;
        if (stage < 4) {
          nu = caxpy(stage == 3 ? hh : h2, k, S.v0[pi]);
          S.v1[pi] = stage == 1 ? k : caxpy((T)2, k, S.v1[pi]);
        } else {
          C cv = S.v2[pi];
          nu = update(S.v1[pi], k, S.v0[pi], cv);
          S.v2[pi] = cv;
          S.v0[pi] = nu;
        }
        S.v3[pi] = nu;
        if (send && lane < len) {
          const int i = xidx(S.pc[q]);
          slot_put(out + slot_of<C>(i), nu, no + 1);
          if (A.rec) (stage < 4 ? recorded(step, stage + 1) : recorded(step + 1, 1))[i] = nu;
        }
      }
      }
      ++no;
      in = out;
    }
  }
  __syncthreads();
  if (*(volatile int*)&dead) return;
  if (SMALL && warp < cta.n) {
    S.v0[32 * warp + lane] = y1;
    S.v2[32 * warp + lane] = c1;
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
// stage exchanged through the numbered slots.  The transposed separable source needs, at a
// point of G, sums over a row or column of b_R: a warp per G point waits for those elements and sums
// them directly, beside the points of R (no reduction phase of its own).  Parameter sums stay in
// registers: per pair u P^T b and u Q^T b, reduced into the gradient slots when an envelope changes
// its value and at the end.
// ONE (at most two pairs, two sandwich terms, eight pieces a CTA and ten row values a lane): a warp's one piece with its
// offsets and state in registers and every value it needs in one batch of loads.
template <typename T, int NP, int THREADS, bool ONE>
__global__ void __launch_bounds__(THREADS, 1) k_grid_adj(const GridArgs A) {
  using C = typename C2T<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[THREADS / 32][2 * NP + BQ_GRID_MAXT + 2];
  __shared__ int segs[2 * 8 * BQ_GRID_MAXP];
  __shared__ GridProb P;
  __shared__ int dead;
  const GridCta cta = A.ctas[blockIdx.x];
  for (int i = threadIdx.x; i < (int)(sizeof(GridProb) / 4); i += THREADS)
    reinterpret_cast<int*>(&P)[i] = reinterpret_cast<const int*>(A.probs + cta.prob)[i];
  if (threadIdx.x == 0) dead = 0;
  __syncthreads();
  const int ng = P.ng, np = P.np, ns = P.ns, nt = P.nt;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = THREADS / 32;
  const int wrow = 4 * np + ns + 2 * nt;  // weights of the row values (ONE)
  const GridSlots<T> S(smem_raw, cta.n, wrow + (ONE ? BQ_GRID_ROWS : 0), 4 * np + ns);
  const int n = S.n;
  C* const E = S.E;
  // weights of the sandwich terms over the flat index (the sums over rows and columns of b_R)
  T* swt = reinterpret_cast<T*>(S.fl + n);
  const C zero = cmk<C>(0.0, 0.0);
  for (int i = tid; i < cta.n * (int)(sizeof(GridPiece) / 4); i += THREADS)
    reinterpret_cast<int*>(S.pc)[i] = reinterpret_cast<const int*>(A.pieces + cta.p0)[i];
  const GridTab<T> W(P, reinterpret_cast<const T*>(A.tab) + P.tab);
  for (int i = tid; i < 2 * ns * ng; i += THREADS) swt[i] = W.sand(0, 0)[i];
  __syncthreads();
  uint4* const ring = reinterpret_cast<uint4*>(A.ring);
  const size_t place = A.place;
  const int places = (int)min((long long)A.ring_places, 4LL * A.n_steps + 1);  // that this launch uses
  auto xidx = [&](const GridPiece& g) {
    return (g.kind <= GRID_D ? g.off_r : g.kind == GRID_X ? g.off_gx : g.off_gy) + g.start + lane;
  };
  int hre_any = 0;
  const T hh = (T)A.dt, w6 = hh * (T)(1.0 / 6.0), w3 = hh * (T)(1.0 / 3.0), h2 = hh * (T)0.5;
  for (int q = warp; q < cta.n; q += nw) {
    const GridPiece g = S.pc[q];
    const int pi = 32 * q + lane;
    const bool ok = lane < g.len;
    const int self = xidx(g), si = ok ? self : self - lane, i = g.start + lane;
    const int k = g.kind == GRID_R ? i / ng : i, l = g.kind == GRID_R ? i - k * ng : i;
    for (int j = 0; j < 4 * np + ns; ++j) {
      S.off[j * n + pi] = slot_of<C>(si);
      S.w[j * n + pi] = (T)0;
    }
    for (int t = 0; t < 2 * nt; ++t) S.w[(4 * np + ns + t) * n + pi] = (T)0;
    C v = zero, dg = zero;
    if (ok) {
      v = reinterpret_cast<const C*>(A.lam)[self];
      for (int r = 0; r < places; ++r)
        if (r != 1) slot_put(ring + r * place + slot_of<C>(self), zero, 0u);
      slot_put(ring + place + slot_of<C>(self), cscale(v, w6), 1u);
      if (g.kind <= GRID_D) dg = W.diag(k, l);
      else if (g.kind == GRID_X) dg = W.diag(0, k, g.c_re, g.c_im);
      else dg = W.diag(1, k, -g.c_re, -g.c_im);
      auto put = [&](int j, T w, int o) {
        if (w == (T)0) return;
        S.w[j * n + pi] = w;
        S.off[j * n + pi] = slot_of<C>(o);
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
        if (h.x != (T)0) hre_any = 1;
        S.w[(4 * np + ns + 2 * t) * n + pi] = h.x;
        S.w[(4 * np + ns + 2 * t + 1) * n + pi] = h.y;
      }
    }
    S.v0[pi] = S.v1[pi] = v;
    S.v3[pi] = cscale(v, w6);
    S.dg[pi] = dg;
    unsigned int any = 0u;
    for (int s = 0; s < ns; ++s)
      if (__any_sync(0xffffffffu, S.w[(4 * np + s) * n + pi] != (T)0)) any |= 1u << s;
    if (lane == 0) S.pc[q].pad = (int)any;
  }
  // parameter sums of this thread: per pair Re sum u (a - b) and Im sum u (a + b), which are all
  // that Re(da S_a - conj(da) S_b) needs
  double gx[NP], gy[NP];
  double2 dcs = make_double2(0.0, 0.0);
  double gt[BQ_GRID_MAXT];
#pragma unroll
  for (int j = 0; j < NP; ++j) gx[j] = gy[j] = 0.0;
#pragma unroll
  for (int t = 0; t < BQ_GRID_MAXT; ++t) gt[t] = 0.0;
  const long long last = A.n_steps - 1;
  // Both halves of the table: the first step may be the lowest of its eight, whose last stage already
  // asks for the segment of the step below, and no block boundary lies between.
  if (warp == nw - 1) {
    grid_envelope<T>(A, P, E, last & ~7LL, segs);
    if (last > 7) grid_envelope<T>(A, P, E, (last & ~7LL) - 8, segs);
  }
  unsigned int block = 0;
  const bool hre = __syncthreads_or(hre_any);
  if (!grid_sync(A.bar, A.error)) return;

  auto seg_of = [&](long long i, int j) { return segs[(((i >> 3) & 1) * 8 + (i & 7)) * BQ_GRID_MAXP + j]; };

  unsigned int no = 1;
  const uint4* in = ring + place;
  int turn = 1;
  // value of pair j at this point: a from sources x.lo, y.lo, b from x.hi, y.hi (see pair_sum)
  int of[ONE ? 14 : 1], go[ONE ? BQ_GRID_ROWS : 1];
  unsigned int on = 0u;
  C l1 = zero, a1 = zero, b1 = zero, dg1 = zero;
  int kind1 = 0, xi1 = -1, xs1 = 0, rows = 0;
  if (ONE && warp < cta.n) {
    const GridPiece& g = S.pc[warp];
    const int pi = 32 * warp + lane;
    const bool isx = g.kind == GRID_X;
    const int self = lane < g.len ? xidx(g) : xidx(g) - lane;  // (for values that a point lacks)
    kind1 = g.kind;
    if (lane < g.len) xi1 = self;
    xs1 = slot_of<C>(self);
    l1 = a1 = S.v0[pi];
    b1 = S.v3[pi];
    dg1 = S.dg[pi];
    if (kind1 <= GRID_D) {  // values 0..7: pairs, 8, 9: sandwich terms
#pragma unroll
      for (int i = 0; i < (ONE ? 14 : 1); ++i) {
        const bool want = i < 8 ? i < 4 * np && kind1 == GRID_R : (unsigned int)g.pad >> (i - 8) & 1u;
        of[i] = want ? S.off[(i < 8 ? i : 4 * np + i - 8) * n + pi] : xs1;
        on |= (want ? 1u : 0u) << i;
      }
    } else {  // values 0..3: lo and hi of the pairs, 4..13: elements of the rows or columns of b_R
      const int nj = P.r_diag ? 1 : (ng + 31) / 32;
      rows = P.has_r ? ns * nj : 0;
#pragma unroll
      for (int i = 0; i < (ONE ? 14 : 1); ++i) {
        of[i] = xs1;
        if (i < 4) {
          if (i < 2 * np && xi1 >= 0) {
            of[i] = S.off[(4 * (i >> 1) + (i & 1)) * n + pi];
            on |= 1u << i;
          }
          continue;
        }
        const int t = i - 4;
        go[t] = 0;
        T wt = (T)0;
        if (t < rows) {
          const int s = t / nj, kk = g.start - P.ss[s], j = P.r_diag ? kk : lane + 32 * (t - s * nj);
          if (kk >= 0 && kk < ng && j < ng && !(P.r_diag && lane)) {
            wt = swt[(2 * s + (isx ? 0 : 1)) * ng + kk] * swt[(2 * s + (isx ? 1 : 0)) * ng + j];
            if (!P.r_diag && P.sst[s] && (j / P.sst[s]) % P.sM[s] != (kk / P.sst[s]) % P.sM[s]) wt = (T)0;
          }
          if (wt != (T)0) {
            of[i] = slot_of<C>(g.off_r + (P.r_diag ? kk : isx ? kk * ng + j : j * ng + kk));
            go[t] = (isx ? g.off_gy : g.off_gx) + P.ss[s] + j;
            on |= 1u << i;
          }
          S.w[(wrow + t) * n + pi] = wt;
        }
      }
    }
  }
  // which sums pair j needs (bits 2 j, 2 j + 1: gy, gx): a static imaginary derivative only Im
  unsigned int gneed = 0u;
  for (int j = 0; j < np; ++j)
    if (P.gpar[j] >= 0 || P.gpwc[j] >= 0)
      gneed |= (P.gpwc[j] >= 0 || P.ch[j] >= 0 || P.cb_re[j] != 0.0 ? 3u : 1u) << (2 * j);
  // q += av a - conj(av) b; s = a + b, d = a - b (where needed)
  auto pair_q = [&](int j, C av, C a, C b, C& s, C& d, C& qv) {
    s = cadd(a, b);
    const bool im = zero_bits(av.x);
    d = zero;
    if (!im || (gneed >> (2 * j) & 2u)) {
      d.x = a.x - b.x;
      d.y = a.y - b.y;
    }
    qv.x = fma(-av.y, s.y, qv.x);
    qv.y = fma(av.y, s.x, qv.y);
    if (!im) {
      qv.x = fma(av.x, d.x, qv.x);
      qv.y = fma(av.x, d.y, qv.y);
    }
  };
  auto pair_sums = [&](int j, C u, C s, C d) {
#pragma unroll
    for (int i = 0; i < NP; ++i)
      if (i == j) {
        if (gneed >> (2 * i) & 1u) grad_add(gy[i], u.x, s.y, u.y, s.x);
        if (gneed >> (2 * i) & 2u) grad_add(gx[i], u.x, d.x, -u.y, d.y);
      }
  };
  auto pair_grad = [&](int j, C av, C a, C b, C u, C& qv) {
    C s, d;
    pair_q(j, av, a, b, s, d, qv);
    pair_sums(j, u, s, d);
  };
  // u b dD/dtheta of the parameters on diagonal terms; their weights are imaginary unless hre
  auto diag_grad = [&](const T* w, C u, C b) {
    const T zy = fma(u.x, b.y, u.y * b.x);
    const T zx = hre ? fma(u.x, b.x, -u.y * b.y) : (T)0;
#pragma unroll
    for (int t = 0; t < BQ_GRID_MAXT; ++t)
      if (t < nt) {
        const T hy = w[(4 * np + ns + 2 * t + 1) * n];
        if (hre) grad_add(gt[t], zx, w[(4 * np + ns + 2 * t) * n], -zy, hy);
        else grad_add(gt[t], -zy, hy);
      }
  };

#pragma unroll 1
  for (long long it = last; it >= 0; --it) {
    if (it != last && ((it + 1) & (A.block - 1)) == 0) {
      if (!block_sync(A.bar, ++block, A.error, &dead)) return;
    }
    // The eight steps below this batch replace those above it, in its first step: the block boundary just
    // passed ended the reads of the upper batch, and the boundary after the batch's first four steps (blocks
    // are of four steps at most) comes before the first read, of a segment in its last step.
    if ((it & 7) == 7 && it != last && it > 7 && warp == nw - 1) grid_envelope<T>(A, P, E, (it & ~7LL) - 8, segs);
#pragma unroll 1
    for (int stage = 4; stage >= 1; --stage) {
      turn = turn + 1 == A.ring_places ? 0 : turn + 1;
      uint4* out = ring + turn * place;
      const C* U = reinterpret_cast<const C*>(A.rec + ((size_t)it * 4 + stage - 1) * A.arr);
      const C* Es = E + (((it >> 3) & 1) * 32 + (it & 7) * 4 + stage - 1) * BQ_GRID_MAXP;
      if constexpr (ONE) {
        if (warp < cta.n) {
          const T* w = S.w + 32 * warp + lane;
          const C u = xi1 >= 0 ? U[xi1] : zero;
          C h[BQ_GRID_ROWS];
          if (kind1 >= GRID_X) {
#pragma unroll
            for (int t = 0; t < BQ_GRID_ROWS; ++t)
              if (t < rows) h[t] = on >> (4 + t) & 1u ? cscale(U[go[t]], w[(wrow + t) * n]) : zero;
          }
          C v[14];
          slots_wait<14>(in, [&](int i) { return of[i]; }, 0xffffffffu, no, v, A.error, &dead);
          // (the gradient sums follow the store: no other warp waits for them)
          C qv = cmul(dg1, b1), ps[2] = {zero, zero}, pd[2] = {zero, zero};
          if (kind1 <= GRID_D) {
#pragma unroll
            for (int j = 0; j < 2; ++j)
              if (on >> (4 * j) & 1u) {
                const T w0 = w[(4 * j) * n], w1 = w[(4 * j + 1) * n], w2 = w[(4 * j + 2) * n], w3_ = w[(4 * j + 3) * n];
                C a, c;
                a.x = fma(w0, v[4 * j].x, -w3_ * v[4 * j + 3].x);
                a.y = fma(w0, v[4 * j].y, -w3_ * v[4 * j + 3].y);
                c.x = fma(w1, v[4 * j + 1].x, -w2 * v[4 * j + 2].x);
                c.y = fma(w1, v[4 * j + 1].y, -w2 * v[4 * j + 2].y);
                pair_q(j, Es[j], a, c, ps[j], pd[j], qv);
              }
#pragma unroll
            for (int s = 0; s < 2; ++s)
              if (on >> (8 + s) & 1u) qv = caxpy(w[(4 * np + s) * n], v[8 + s], qv);
          } else {
            const bool isx = kind1 == GRID_X;
            C r0 = zero, r1 = zero;
#pragma unroll
            for (int t = 0; t < BQ_GRID_ROWS; ++t)
              if (t < rows) {
                if (t & 1) r1 = cfma(v[4 + t], h[t], r1);
                else r0 = cfma(v[4 + t], h[t], r0);
              }
            r0 = cadd(r0, r1);
            // lanes 0..15 sum the real parts, 16..31 the imaginary ones
            const bool up = lane & 16;
            T x = up ? r0.y : r0.x;
            x += __shfl_xor_sync(0xffffffffu, up ? r0.x : r0.y, 16);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            const T xi = __shfl_sync(0xffffffffu, x, 16);
            if (lane == 0) {
              qv.x += x;
              qv.y += xi;
            }
            // (lanes without a point hold zeros throughout)
#pragma unroll
            for (int j = 0; j < 2; ++j)
              if (j < np) {
                const C lo = cscale(v[2 * j], w[(4 * j) * n]), hi = cscale(v[2 * j + 1], w[(4 * j + 1) * n]);
                // X: a lo - conj(a) hi;  Y: conj(a) lo - a hi = a (-hi) - conj(a) (-lo)
                pair_q(j, Es[j], isx ? lo : cneg(hi), isx ? hi : cneg(lo), ps[j], pd[j], qv);
              }
          }
          const C b0 = b1;
          a1 = cadd(a1, qv);  // (the step's sum starts as lam)
          if (stage > 1) {
            b1 = caxpy(stage == 4 ? hh : h2, qv, cscale(l1, stage == 2 ? w6 : w3));
          } else {
            l1 = a1;
            b1 = cscale(a1, w6);
          }
          if (xi1 >= 0 && (it > 0 || stage > 1)) slot_put(out + xs1, b1, no + 1);
#pragma unroll
          for (int j = 0; j < 2; ++j)
            if (j < np) pair_sums(j, u, ps[j], pd[j]);
          if (nt) diag_grad(w, u, b0);
          if (kind1 >= GRID_X) {
            const C z = cmul(u, b0);
            if (kind1 == GRID_X) dcs = make_double2(dcs.x + (double)z.x, dcs.y + (double)z.y);
            else dcs = make_double2(dcs.x - (double)z.x, dcs.y - (double)z.y);
          }
        }
      } else {
#pragma unroll 1
      for (int q = warp; q < cta.n; q += nw) {
        const GridPiece& g = S.pc[q];
        const int kind = g.kind, len = g.len;
        const unsigned int any = (unsigned int)g.pad;
        const int pi = 32 * q + lane;
        const T* w = S.w + pi;
        const int* off = S.off + pi;
        const C b = S.v3[pi];
        const bool ok = lane < len;
        const C u = ok ? U[xidx(g)] : zero;
        C qv = cmul(S.dg[pi], b);
        if (kind == GRID_R) {
          C sv[4];
          auto pair = [&](int j, C n0, C n1, C n2, C n3) {
            const T w0 = w[(4 * j) * n], w1 = w[(4 * j + 1) * n], w2 = w[(4 * j + 2) * n], w3_ = w[(4 * j + 3) * n];
            C a, c;
            a.x = fma(w0, n0.x, -w3_ * n3.x);
            a.y = fma(w0, n0.y, -w3_ * n3.y);
            c.x = fma(w1, n1.x, -w2 * n2.x);
            c.y = fma(w1, n1.y, -w2 * n2.y);
            pair_grad(j, Es[j], a, c, u, qv);
          };
#pragma unroll 1
            for (int j0 = 0; j0 < np; j0 += 2) {
              const int m = min(2, np - j0);
              C v[8];
              slots_wait<8>(in, [&](int i) { return off[(4 * j0 + i) * n]; }, (1u << (4 * m)) - 1u, no, v, A.error, &dead);
#pragma unroll
              for (int i = 0; i < 2; ++i)
                if (i < m) pair(j0 + i, v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            }
            slots_wait<4>(in, [&](int i) { return off[(4 * np + i) * n]; }, any, no, sv, A.error, &dead);
#pragma unroll
          for (int s = 0; s < 4; ++s)
            if (any >> s & 1u) qv = caxpy(w[(4 * np + s) * n], sv[s], qv);
        } else if (kind == GRID_D) {
          C sv[4];
          slots_wait<4>(in, [&](int i) { return off[(4 * np + i) * n]; }, any, no, sv, A.error, &dead);
#pragma unroll
          for (int s = 0; s < 4; ++s)
            if (any >> s & 1u) qv = caxpy(w[(4 * np + s) * n], sv[s], qv);
        } else {
          // a point of G, the whole warp on it: the transposed source's sum over a row (G_x) or column
          // (G_y) of b_R, then the point's own lane the rest
          const bool isx = kind == GRID_X;
          C src = zero;
          if (P.has_r) {
            for (int s = 0; s < ns; ++s) {
              const int kk = g.start - P.ss[s];  // row / column of b_R
              if (kk < 0 || kk >= ng) continue;
              const T wt = swt[(2 * s + (isx ? 0 : 1)) * ng + kk];
              if (wt == (T)0) continue;
              const T* wo = swt + (2 * s + (isx ? 1 : 0)) * ng;
              const C* go = U + (isx ? g.off_gy : g.off_gx) + P.ss[s];
              C v = zero;
              if (P.r_diag) {
                const T wj = lane == 0 ? wo[kk] : (T)0;  // (the whole warp calls slots_wait)
                C x[1];
                slots_wait<1>(in, [&](int) { return slot_of<C>(g.off_r + kk); }, wj != (T)0 ? 1u : 0u, no, x, A.error, &dead);
                if (wj != (T)0) v = cmul(x[0], cscale(go[kk], wj));
              } else {
                const int mk = P.sst[s] ? (kk / P.sst[s]) % P.sM[s] : 0;
                const int br = g.off_r + (isx ? kk * ng : kk), st = isx ? 1 : ng;
#pragma unroll 1
                for (int jb = 0; jb < ng; jb += 192) {
                  const int j0 = jb + lane;
                  unsigned int on = 0u;
                  C x[6];
#pragma unroll
                  for (int i = 0; i < 6; ++i) {
                    const int j = j0 + 32 * i;
                    if (j < ng && wo[j] != (T)0 && !(P.sst[s] && (j / P.sst[s]) % P.sM[s] != mk)) on |= 1u << i;
                  }
                  slots_wait<6>(in, [&](int i) { return slot_of<C>(br + (j0 + 32 * i) * st); }, on, no, x, A.error, &dead);
#pragma unroll
                  for (int i = 0; i < 6; ++i)
                    if (on >> i & 1u) v = cfma(x[i], cscale(go[j0 + 32 * i], wo[j0 + 32 * i]), v);
                }
              }
              src = caxpy(wt, v, src);
            }
            __syncwarp();
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
              src.x += __shfl_xor_sync(0xffffffffu, src.x, o);
              src.y += __shfl_xor_sync(0xffffffffu, src.y, o);
            }
          }
          if (ok) qv = cadd(qv, src);
#pragma unroll 1
          for (int j0 = 0; j0 < np; j0 += 2) {
            const int m = min(2, np - j0);
            C v[4];
            slots_wait<4>(in, [&](int i) { return off[(4 * (j0 + i / 2) + (i & 1)) * n]; },
                          ok ? (1u << (2 * m)) - 1u : 0u, no, v, A.error, &dead);
            if (ok) {
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                if (i >= m) break;
                const int j = j0 + i;
                const C lo = cscale(v[2 * i], w[(4 * j) * n]), hi = cscale(v[2 * i + 1], w[(4 * j + 1) * n]);
                // X: a lo - conj(a) hi;  Y: conj(a) lo - a hi = a (-hi) - conj(a) (-lo)
                pair_grad(j, Es[j], isx ? lo : cneg(hi), isx ? hi : cneg(lo), u, qv);
              }
            }
          }
          if (ok) {
            const C z = cmul(u, b);
            if (isx) dcs = make_double2(dcs.x + (double)z.x, dcs.y + (double)z.y);
            else dcs = make_double2(dcs.x - (double)z.x, dcs.y - (double)z.y);
          }
          __syncwarp();
        }
        if (nt) diag_grad(w, u, b);
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
          if (it > 0 || stage > 1) slot_put(out + slot_of<C>(xidx(g)), bn, no + 1);
        }
      }
      }
      ++no;
      in = out;
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
          const double x = sum(gx[j]), y = sum(gy[j]);
          if (lane == 0) {
            red[warp][2 * j] = x;
            red[warp][2 * j + 1] = y;
          }
          gx[j] = gy[j] = 0.0;
        }
#pragma unroll
        for (int t = 0; t < BQ_GRID_MAXT; ++t) {
          if (t >= nt) break;
          const double x = sum(gt[t]);
          if (lane == 0) red[warp][2 * NP + t] = x;
          gt[t] = 0.0;
        }
        {
          const double x = sum(dcs.x), y = sum(dcs.y);
          if (lane == 0) {
            red[warp][2 * NP + BQ_GRID_MAXT] = x;
            red[warp][2 * NP + BQ_GRID_MAXT + 1] = y;
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
          const double x = col(2 * j), y = col(2 * j + 1);
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
          auto dre = [&](double2 da) { return da.x * x - da.y * y; };
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
        if (tid >= 32 && tid < 32 + nt) atomicAdd(A.grad + P.tpar[tid - 32], col(2 * NP + tid - 32));
        __syncthreads();
        // the separation constant's dependence on the parameters (an adjoint CTA holds one system)
        if (P.has_sep) {
          const double x = col(2 * NP + BQ_GRID_MAXT), y = col(2 * NP + BQ_GRID_MAXT + 1);
          for (int i = tid; i < P.n_params; i += THREADS) {
            const double2 v = A.dc[S.pc[0].dc_off + i];
            if (v.x != 0.0 || v.y != 0.0) atomicAdd(A.grad + P.grad_off + i, v.x * x - v.y * y);
          }
        }
        __syncthreads();
      }
    }
  }
  __syncthreads();
  if (*(volatile int*)&dead) return;
  if (ONE && warp < cta.n) S.v0[32 * warp + lane] = l1;
  for (int q = warp; q < cta.n; q += nw) {
    const GridPiece& g = S.pc[q];
    if (lane < g.len) reinterpret_cast<C*>(A.lam)[xidx(g)] = S.v0[32 * q + lane];
  }
}

template <typename T>
static const void* grid_func_t(int np, int ns, bool adj, int form) {
  if (adj) {
    if (form == GRID_ONE) return (const void*)k_grid_adj<T, 2, 256, true>;
    if (np <= 2) return form == GRID_FEW ? (const void*)k_grid_adj<T, 2, 256, false> : (const void*)k_grid_adj<T, 2, 512, false>;
    if (np <= 4) return form == GRID_FEW ? (const void*)k_grid_adj<T, 4, 256, false> : (const void*)k_grid_adj<T, 4, 512, false>;
    return nullptr;
  }
  if (form == GRID_ONE)
    return np > 1 ? (const void*)k_grid_fwd<T, 2, 2, 256> : ns > 1 ? (const void*)k_grid_fwd<T, 1, 2, 256> : (const void*)k_grid_fwd<T, 1, 1, 256>;
  return form == GRID_FEW ? (const void*)k_grid_fwd<T, 0, 0, 256> : (const void*)k_grid_fwd<T, 0, 0, 512>;
}

static cudaError_t launch_grid_any(const void* f, const GridArgs& a, int ctas, int form, int smem_bytes, cudaStream_t s) {
  if (!f || ctas < 1) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, BQ_GRID_SMEM_MAX);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(a.bar, 0, BQ_GRID_BAR_WORDS * sizeof(unsigned int), s);
  if (e != cudaSuccess) return e;
  GridArgs p = a;
  void* args[] = {(void*)&p};
  return cudaLaunchCooperativeKernel(f, dim3(ctas), dim3(grid_threads(form)), args, (size_t)smem_bytes, s);
}

}  // namespace bq
