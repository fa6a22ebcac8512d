// Device helpers shared by the translation units that hold kernels: complex arithmetic on
// float2 / double2, error-free addition, and drive envelopes at the RK4 stage times.
#pragma once

#include <cuda_runtime.h>

#include "bq_internal.h"

namespace bq {

template <typename T> struct C2T;
template <> struct C2T<double> { using type = double2; };
template <> struct C2T<float> { using type = float2; };

template <typename C> __device__ __forceinline__ C cmk(double re, double im);
template <> __device__ __forceinline__ double2 cmk<double2>(double re, double im) { return make_double2(re, im); }
template <> __device__ __forceinline__ float2 cmk<float2>(double re, double im) {
  return make_float2((float)re, (float)im);
}

template <typename C> __device__ __forceinline__ C cadd(C a, C b) { a.x += b.x; a.y += b.y; return a; }
template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
  C r; r.x = a.x * b.x - a.y * b.y; r.y = a.x * b.y + a.y * b.x; return r;
}
// a + s * b (complex s)
template <typename C> __device__ __forceinline__ C cfma(C s, C b, C a) {
  a.x = fma(s.x, b.x, fma(-s.y, b.y, a.x));
  a.y = fma(s.x, b.y, fma(s.y, b.x, a.y));
  return a;
}
template <typename C, typename T> __device__ __forceinline__ C cscale(C a, T s) { a.x *= s; a.y *= s; return a; }
// a + s * b (real s)
template <typename C, typename T> __device__ __forceinline__ C caxpy(T s, C b, C a) {
  a.x = fma(s, b.x, a.x); a.y = fma(s, b.y, a.y); return a;
}

__device__ __forceinline__ double stage_c(int stage) {
  return stage == 1 ? 0.0 : (stage == 4 ? 1.0 : 0.5);
}

template <typename T> __device__ __forceinline__ T dev_exp(T x);
template <> __device__ __forceinline__ double dev_exp<double>(double x) { return exp(x); }
template <> __device__ __forceinline__ float dev_exp<float>(float x) { return expf(x); }

// Physical time of this launch's RK4 stage for a channel of the given kind: the stage time
// tau_step + c_s dt (a piecewise-constant envelope at the step midpoint: the Hamiltonian is
// held constant within a step), mapped to t = horizon - tau for the reversed-time reading.
__device__ __forceinline__ double pipe_chan_time(int kind, double tau_step, int stage, double dt, double horizon,
                                                 int reverse) {
  const double tau = (kind == 2) ? tau_step + 0.5 * dt : tau_step + stage_c(stage) * dt;
  return reverse ? horizon - tau : tau;
}

// Envelope value (bq.h channel kinds) at physical time t (t_mid: the step midpoint, where a
// piecewise-constant envelope is read) from a parameter block's record.  In FP32 the Gaussian
// runs on the FP32 pipe alone (GB300's FP64 rate is a small fraction of its FP32 rate and this
// sits on every system's path): t and the centre come as unevaluated FP32 pairs (t32: hi, lo),
// and t - centre = (t_hi - c_hi) + (t_lo - c_lo), where the first difference is exact wherever
// the pulse is not negligible (Sterbenz: t within a factor 2 of the centre) and elsewhere off
// by at most half an ulp of the centre.  A piecewise-constant envelope reads its segment value
// from the channel parameter pool.
template <typename T>
__device__ __forceinline__ typename C2T<T>::type pipe_chan_value(const PipeChan& c, const double* chpar, double t,
                                                                 double t_mid, const float (&t32)[2]) {
  using C = typename C2T<T>::type;
  switch (c.kind) {
    case 0:  // CONST
      return cmk<C>(c.p[0], c.p[1]);
    case 1: {  // GAUSS
      C v;
      if constexpr (sizeof(T) == 8) {
        const double d = t - c.p[2];
        const double e = dev_exp<double>(-(d * d) / (2.0 * c.p[3] * c.p[3]));
        v.x = c.p[0] * e;
        v.y = c.p[1] * e;
      } else {
        const float d = (t32[0] - c.f[3]) + (t32[1] - c.c_lo);
        const float e = dev_exp<float>(-(d * d) * c.f[2]);
        v.x = c.f[0] * e;
        v.y = c.f[1] * e;
      }
      return v;
    }
    case 2: {  // PWC
      const int n_seg = (c.n_par - 2) / 2;
      const double x = floor((t_mid - c.p[0]) / c.p[1]);
      if (!(x >= 0.0) || x >= (double)n_seg) return cmk<C>(0.0, 0.0);
      const int sg = (int)x;
      return cmk<C>(chpar[c.par_off + 2 + 2 * sg], chpar[c.par_off + 3 + 2 * sg]);
    }
    case 3: {  // CEXP
      double sn, cs;
      sincos(c.p[2] * t, &sn, &cs);
      return cmk<C>(c.p[0] * cs - c.p[1] * sn, c.p[0] * sn + c.p[1] * cs);
    }
    default:
      return cmk<C>(0.0, 0.0);
  }
}

// Error-free sum of two complex values componentwise (Knuth's TwoSum, no magnitude
// condition): s = fl(a + b) and s + e == a + b exactly.
template <typename C>
__device__ __forceinline__ void two_sum(C a, C b, C& s, C& e) {
  s.x = a.x + b.x;
  s.y = a.y + b.y;
  const auto bx = s.x - a.x;
  const auto by = s.y - a.y;
  e.x = (a.x - (s.x - bx)) + (b.x - bx);
  e.y = (a.y - (s.y - by)) + (b.y - by);
}

// The same with half the FP64 instructions: Fast2Sum, which is exact unless the first operand's exponent
// is the smaller one, with the operands put in order by their high words, compared as FP32 values (a
// compare takes the magnitudes for free; it is false only from 2^1016 on).  1024 FP64 oscillators,
// us per step: plain Fast2Sum 118.0, this 120.3, TwoSum 127.6.
__device__ __forceinline__ void sum_ordered(double a, double b, double& s, double& e) {
  const bool swap = fabsf(__int_as_float(__double2hiint(a))) < fabsf(__int_as_float(__double2hiint(b)));
  const double big = swap ? b : a, small = swap ? a : b;
  s = a + b;
  e = small - (s - big);
}
__device__ __forceinline__ void sum_ordered(double2 a, double2 b, double2& s, double2& e) {
  sum_ordered(a.x, b.x, s.x, e.x);
  sum_ordered(a.y, b.y, s.y, e.y);
}
__device__ __forceinline__ void sum_ordered(float2 a, float2 b, float2& s, float2& e) { two_sum(a, b, s, e); }

template <typename C>
__device__ __forceinline__ C cneg(C a) {
  a.x = -a.x;
  a.y = -a.y;
  return a;
}

}  // namespace bq
