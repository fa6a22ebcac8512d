// Grid-resident kernels of the tiled path (k_grid_fwd, k_grid_adj): data structures shared by
// the host plan and the kernels, and the host-side launchers.
#pragma once

#include <cuda_runtime.h>

#include "bq_internal.h"

#define BQ_GRID_MAX_CTAS 152  // one per SM of a GB300
#define BQ_GRID_MAXP 8   // off-diagonal pairs of a problem
#define BQ_GRID_MAXS 4   // sandwich terms
#define BQ_GRID_MAXT 4   // parameters that multiply diagonal terms
#define BQ_GRID_SMEM_MAX (200 * 1024)
#define BQ_GRID_ROWS 10   // row values a lane of an adjoint piece of G may need (GRID_ONE)
#define BQ_GRID_BAR_WORDS 5

namespace bq {

// Per-problem tables, element type of the state, n_g entries each, from element offset tab (in
// reals): dx, dy, then what they lack of the exact sums (complex), then per pair xm xp ym yp (real), per sandwich term sx sy (real);
// for the adjoint the same weights at the transposed sources: per pair xmT xpT ymT ypT, per
// sandwich term sxT syT; per diagonal parameter hx hy (complex).
struct GridProb {
  int ng, np, ns, nt;
  int has_sep, has_r, r_diag, herm;
  long long tab;
  int dlt[BQ_GRID_MAXP];      // pair j: X sources k - dlt (coefficient a) and k + dlt (-conj a), Y
                              // sources l + dlt (-a) and l - dlt (conj a)
  int ch[BQ_GRID_MAXP], cj[BQ_GRID_MAXP];  // envelope (index below, -1: none) and its conjugation in a
  double a_re[BQ_GRID_MAXP], a_im[BQ_GRID_MAXP];
  double cb_re[BQ_GRID_MAXP], cb_im[BQ_GRID_MAXP];  // a's static part with its parameter set to 1
  int gpar[BQ_GRID_MAXP], gpwc[BQ_GRID_MAXP];       // gradient slots (-1: none)
  int ss[BQ_GRID_MAXS];       // sandwich term q: source (k + ss, l + ss)
  int sst[BQ_GRID_MAXS], sM[BQ_GRID_MAXS];  // restricted to equal indices (k / sst) % sM (sst 0: everywhere)
  int tpar[BQ_GRID_MAXT];     // gradient slots of the diagonal parameters
  int nch, n_params, grad_off, pad;
  ChanDesc cd[BQ_GRID_MAXP];
  PipeChan chan[BQ_GRID_MAXP];
};

enum GridKind : int { GRID_R = 0, GRID_H = 1, GRID_D = 2, GRID_X = 3, GRID_Y = 4 };

// Up to 32 points of one kind of one system, one per lane (the adjoint: a point of G is a piece, a warp
// sums its row or column).  start: first point in the kind's own numbering.
struct GridPiece {
  int sys, kind, start, len;
  int off_gx, off_gy, off_r, pad;
  double c_re, c_im;  // separation constant
  int dc_off, pad2[3];
};
struct GridCta {
  int prob, p0, n, pad;  // pieces [p0, p0 + n)
};

struct GridArgs {
  const GridCta* ctas;
  const GridPiece* pieces;
  const GridProb* probs;
  const void* tab;
  const double* chpar;
  void* y;
  void* comp;
  void* ring;     // exchange of stage inputs (adjoint: of b): ring_places x place 16-byte words
  size_t place;   // grid_place()
  int ring_places, block;  // places; steps (a power of two) between the CTAs' block counts
  char* rec;      // recorded stage inputs (4 per step) or null
  size_t arr;     // bytes of one state array
  unsigned int* bar;    // BQ_GRID_BAR_WORDS counters, zeroed before the launch
  unsigned int* error;  // bit 2 is set when a barrier wait gives up
  void* lam;      // adjoint: cotangent of the state, in and out
  double* grad;
  const double2* dc;
  int comp_zero, reverse, n_steps;
  int single_mode;  // FP64: the state update is error-free whatever the increment (as in the single-mode kernels)
  int herm;       // the pieces hold the Hermitian problems in the Hermitian layout
  long long step0;      // the first step is at tau0 + step0 dt
  double dt, tau0, horizon;
};

// Largest grid whose CTAs are all resident (0: no cooperative launch), and the launches.
cudaError_t grid_max_ctas(int dtype, int np, int ns, bool adj, int form, int smem_bytes, int* out);
cudaError_t launch_grid_f32(const GridArgs& a, int np, int ns, bool adj, int ctas, int form, int smem_bytes, cudaStream_t s);
cudaError_t launch_grid_f64(const GridArgs& a, int np, int ns, bool adj, int ctas, int form, int smem_bytes, cudaStream_t s);
const void* grid_func_f32(int np, int ns, bool adj, int form);
const void* grid_func_f64(int np, int ns, bool adj, int form);

// 16-byte words of a place of the ring: a state's slots, in whole groups of 32 (FP64: two words each).
inline size_t grid_place(size_t elems, size_t cs) { return (elems + 31) / 32 * (cs == 16 ? 64 : 32); }
// Forms of the kernels, by the largest number n of pieces in a CTA: a piece per warp in registers (small
// problems), eight warps, sixteen warps.
enum GridForm : int { GRID_ONE = 0, GRID_FEW = 1, GRID_MANY = 2 };
inline int grid_threads(int form) { return form == GRID_MANY ? 512 : 256; }
// Whether a problem is small enough for GRID_ONE.
inline bool grid_small(const GridProb& p, bool adj) {
  return p.np <= 2 && p.ns <= 2 && (!adj || !p.has_r || p.r_diag || p.ns * ((p.ng + 31) / 32) <= BQ_GRID_ROWS);
}

// Dynamic shared memory of a CTA with n pieces (cs: complex size): per point five complex values,
// the weights, the offsets and a flag word; envelopes; in the adjoint the sandwich tables.
inline size_t grid_smem(int n, const GridProb& p, bool adj, int form, size_t cs) {
  const int nw = 4 * p.np + p.ns + (adj ? 2 * p.nt + (form == GRID_ONE ? BQ_GRID_ROWS : 0) : 0), no = 4 * p.np + (adj ? 1 : 3) * p.ns;
  return (size_t)n * sizeof(GridPiece) + (size_t)n * 32 * (5 * cs + nw * (cs / 2) + (no + 1) * 4) +
         (size_t)2 * 32 * BQ_GRID_MAXP * cs + (adj ? (size_t)2 * p.ns * p.ng * (cs / 2) : 0) + 16;
}

}  // namespace bq
