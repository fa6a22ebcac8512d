// Resident single-mode kernel (k_resident): data structures shared by the host plan and the
// kernel, and the host-side launchers.
#pragma once

#include <cuda_runtime.h>

#include "bq_internal.h"

// warps of a CTA: FP32 two CTAs per SM (128 registers a thread; 112 in the general layout, whose
// largest systems take nine warps), FP64 one
#define BQ_RES_WARPS(cs, herm) ((cs) == 16 ? 16 : (herm) ? 10 : 9)
#define BQ_RES_MAXW 16
// elements from one row of a stage buffer to the next (P <= 43)
#define BQ_RES_COLS 44
#define BQ_RES_SMEM_MAX (200 * 1024)

namespace bq {

// One system as a group of warps of a CTA integrates it: nwarps - 1 warps of strips, then one
// warp for G_x, G_y and the drive envelope.
struct ResGroup {
  int sys;        // system index (observable, Hermitian flag)
  int M;          // grid size
  int blk_off;    // element offset of the system block [G_x | G_y | R] in the state arrays
  int blk_elems;  // its length (multiple of 4)
  int gy_off, r_off;  // element offsets inside the block (gy_off -1: no separable part)
  int param_off;  // byte offset of the problem's parameter block (ResHdr)
  int rb, nb;     // rows of a strip, strips per column
  int nwarps;     // warps of the group
  int warp0;      // first warp in the CTA
  int smem_off;   // byte offset of the group's shared memory
  int stage_elems;  // complex elements of the stage buffers (and of the load / store staging)
  int pad;
  double c_re, c_im;  // separation constant C (Eq. 304)
  double w_re, w_im;  // weight of the initial condition
};

// The groups of a CTA: group index of every warp (-1: idle warp).
struct ResBin {
  int g[BQ_RES_MAXW];
};

// Parameter block of a problem: this header, then (element type of the state) dx[M], dy[M]
// (complex), xm, xp, ym, yp, smx, smy, spx, spy (real, M each), then n_obs EvalEntry-like
// records (PipeObs<double2>) at a 16-byte boundary.
//   xm / xp: weights of the left-hand (X) terms with source k - 1 / k + 1, ym / yp: of the
//   right-hand (Y) terms; smx smy / spx spy: row and column weights of the sandwich terms with
//   sources (k - 1, l - 1) / (k + 1, l + 1), their rate folded into the row weight.
struct ResHdr {
  int n_obs, obs_off;  // the observable's entries: count and byte offset
  int ch;             // 1: the off-diagonal terms follow the envelope below
  int conj;           // of the X term with source k - 1
  double a_re, a_im;  // coefficient of the X term with source k - 1 (static part)
  PipeChan chan;
};

struct ResArgs {
  const ResGroup* groups;
  const ResBin* bins;
  const unsigned char* params;
  const double* chpar;
  const unsigned char* flags;  // per system: state is Hermitian (null: not consulted)
  void* y;
  void* comp;
  double2* obs;                // per system w sum_e f_e G(k_e, l_e) of the final state
  int want;                    // with flags: 1 = systems whose flag is set, 0 = the others
  int comp_zero;               // comp is known to be zero and not read
  int reverse;
  int n_steps;
  long long step0;             // the launch's first step is at tau0 + step0 dt
  double dt, tau0, horizon;
  // dt, dt / 2 and the pair w_hi + w_lo = dt / 6 in the state's precision (converted on the host: in
  // the kernel the compiler repeats the conversions every stage, on the scarce FP64 pipe)
  double cd[4];
  float cf[4];
};

// Steps every system of the bins' groups by a.n_steps RK4 steps in one launch; the groups are laid
// out for Hermitian systems (herm) or for any (gen).  variant: bit 0 = the off-diagonal coefficient
// is not purely imaginary at all times, bit 1 = there are sandwich terms with source (k + 1, l + 1),
// bit 2 = the sandwich terms are restricted to k = l.
cudaError_t launch_resident_f32_herm(const ResArgs& a, int variant, int n_bins, int smem_bytes, cudaStream_t s);
cudaError_t launch_resident_f32_gen(const ResArgs& a, int variant, int n_bins, int smem_bytes, cudaStream_t s);
cudaError_t launch_resident_f64_herm(const ResArgs& a, int variant, int n_bins, int smem_bytes, cudaStream_t s);
cudaError_t launch_resident_f64_gen(const ResArgs& a, int variant, int n_bins, int smem_bytes, cudaStream_t s);
// flags[sys] = 1 where the system's G_x, G_y, R (and their compensation) are exactly Hermitian
// (G_y = conj G_x, R = R^dagger) for the n groups given.
cudaError_t launch_res_check(const ResGroup* groups, int n, const void* y, const void* comp, int comp_zero, int dtype,
                             unsigned char* flags, cudaStream_t s);

// Elements from one strip of a stage buffer to the next: its rows, rounded up to P modulo 16.
__host__ __device__ inline int res_strip_stride(int rb, int P) { return rb * BQ_RES_COLS + (((P - rb * BQ_RES_COLS) % 16 + 16) % 16); }
// Shared memory (bytes) of a group: stage buffers, G stage inputs, row products, envelope table.
inline size_t res_group_smem(int stage_elems, int M, size_t cs) {
  const int cols = M | 1;  // (the Hermitian layout's columns)
  return (((size_t)stage_elems + 4 * cols + 8 * cols + 64) * cs + 15) & ~(size_t)15;
}

}  // namespace bq
