// sv_window1d.cuh -- the 1D MUSCL-Hancock step of one warp on a window of cells
// (Sec. 2.3: eqs. 13-15 with xi = 0, source Y, eq. 16 bound), the whole window
// in registers, and the clock of a run that is stepped inside a kernel.
//
// A warp's window holds up to OWN cells that it updates (60 in float, two per
// lane in packed pairs; 28 in double, one per lane) and two halo cells on either
// side, whose slopes, predictors and faces it computes itself: within a step
// lanes exchange only shuffles, and warps nothing.  Per cell the arithmetic is
// that of the step kernels, function for function.
#pragma once

#include "sv_step1d.cuh"

namespace sv {

namespace {

template <typename R> struct Win;
template <> struct Win<float> { static constexpr int CPL = 2, OWN = 60; };
template <> struct Win<double> { static constexpr int CPL = 1, OWN = 28; };

// Maxima over a warp as unsigned keys (one redux instruction per 32 bits).
__device__ __forceinline__ uint32_t fkey(float x) {
  const uint32_t b = __float_as_uint(x);
  return (b >> 31) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float fkey_value(uint32_t k) {
  return __uint_as_float((k >> 31) ? (k & 0x7fffffffu) : ~k);
}
__device__ __forceinline__ float warp_max(float x) {
  return fkey_value(__reduce_max_sync(0xffffffffu, fkey(x)));
}
__device__ __forceinline__ double warp_max(double x) {
  const uint64_t k = key_of(x);
  const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(k >> 32));
  const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(k >> 32) == hi ? (uint32_t)k : 0u);
  return key_to_double(((uint64_t)hi << 32) | lo);
}

// Step size of the run, advanced by every warp alike.  The time itself is kept
// by one warp (`keep`), whose sums nothing waits for: an FP64 operation takes
// a scheduler 64 cycles.  The others hold a float below horizon - t, which says
// that a step cannot be the last one (or reach the next due time); when it does
// not, all warps take the time from shared memory and decide exactly, as the
// per-step finalize does.
template <typename R>
struct Clock {
  double t, t_end;                // t: in the keeping warp; in all after an exact advance
  double horizon;                 // min(t_end, the next time something is due)
  R dt, dt_cfl;                   // of the next step; before the clamp to t_end
  float rest, slack;              // below horizon - t; above t's rounding per step
  uint32_t flags;
  bool last, stop;
  static __device__ __forceinline__ float below(double x) {
    return (float)x * (1.0f - 0x1p-20f);
  }
  // Start at time t0 with the next step d (clamped to t_end: last0).
  __device__ __forceinline__ void start(double t0, double end, R d, bool last0) {
    t = t0;
    t_end = horizon = end;
    dt = d;
    last = last0;
    flags = 0;
    stop = false;
    slack = isfinite(end) ? (float)((fabs(t0) + fabs(end)) * 0x1p-51) : 0.0f;
    rest = below(end - t0);
  }
  // Something is due at time h as well (after an exact advance).
  __device__ __forceinline__ void due(double h) {
    horizon = h < t_end ? h : t_end;
    rest = below(horizon - t);
  }
  // The step of `dt` is complete with these maxima and flags f: the next one's
  // dt.  Called by the whole block, with the same values in every thread;
  // `word` is shared memory; `check`: decide exactly.  Returns whether t is
  // exact in every thread; then `extra(t)` has added its flags.
  template <typename X>
  __device__ __forceinline__ bool advance(const KParams& kp, R smax, R akey, uint32_t f, bool keep,
                                          volatile double* word, bool check, X&& extra) {
    if (keep) t = last ? t_end : t + (double)dt;
    const R d = step_rule(kp, smax, akey, f);
    dt_cfl = d;
    flags = f;
    // the roundings of this and of t stay below the two margins (t_end = inf:
    // rest stays inf)
    rest = fmaf(rest, 1.0f - 0x1p-21f, -(above(dt) + slack));
    dt = d;
    stop = f != 0;
    if (!stop && !last && !check && above(d) < rest) return false;
    // near the horizon, or a flag: exactly
    if (keep && (threadIdx.x & 31) == 0) *word = t;
    __syncthreads();
    t = *word;
    __syncthreads();
    f |= extra(t);
    flags = f;
    last = false;
    stop = f != 0 || !(t < t_end);
    if (stop) {
      dt = (R)0;
    } else {
      const double r = t_end - t;
      rest = below(horizon - t);
      if ((double)d >= r) {
        dt_last = r;
        dt = (R)r;
        last = true;
      }
    }
    return true;
  }
  double dt_last;                 // the last step's dt (t_end - t)
  static __device__ __forceinline__ float above(float x) { return x; }
  // the float at or above a positive double, from its bits; +inf beyond range
  static __device__ __forceinline__ float above(double x) {
    bool ok = true;
    const float v = d64::trunc_f(x, ok);
    return ok ? v * (1.0f + 0x1p-22f) : INFINITY;
  }
};

// One step of a window (float: two per lane).  X: the lane's cells,
// own[]: which of them are updated; folds their bounds.
template <int PP, int LIM, int SRC>
__device__ __forceinline__ void window_step(const P<float>& k, float (&X)[2][4], const bool (&own)[2],
                                         const StepDt<float>& sd, Acc<float>& acc) {
  using pk::f2;
  const f2 dt2 = pk::splat(sd.dt), ndtdx2 = pk::splat(-sd.dtdx);
  const f2 ndt_2h2 = pk::splat(-sd.dt_2h), dt_22 = pk::splat(sd.dt_2);
  f2 U[4], A[4], B[4], WP[4], WM[4], YE, YEv, L[4], F[4], FR[4], Nw[4];
  float xl[4];
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    U[f] = pk::pair(X[0][f], X[1][f]);
    xl[f] = __shfl_up_sync(0xffffffffu, X[1][f], 1);
    const float xr = __shfl_down_sync(0xffffffffu, X[0][f], 1);
    const float c = U[f].y - U[f].x;
    A[f] = pk::pair(U[f].x - xl[f], c);
    B[f] = pk::pair(c, xr - U[f].y);
  }
  pkx::predict<PP, LIM, SRC>(k, U, A, B, ndt_2h2, dt_22, WP, WM, YE, YEv);
#pragma unroll
  for (int f = 0; f < 4; ++f) L[f] = pk::pair(__shfl_up_sync(0xffffffffu, WP[f].y, 1), WP[f].x);
  pkx::hll<PP>(k, L, WM, xl, U, F);
#pragma unroll
  for (int f = 0; f < 4; ++f) FR[f] = pk::pair(F[f].y, __shfl_down_sync(0xffffffffu, F[f].x, 1));
  pk::update<SRC>(U, F, FR, YE, YEv, dt2, ndtdx2, Nw);
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    if (own[0]) X[0][f] = Nw[f].x;
    if (own[1]) X[1][f] = Nw[f].y;
  }
  pkx::cfl<PP, SRC>(k, Nw, (own[0] ? 1 : 0) | (own[1] ? 2 : 0), acc.smax, acc.akey, acc.flags);
}

// The same in double, one cell per lane.
template <int PP, int LIM, int SRC>
__device__ __forceinline__ void window_step(const P<double>& k, double (&X)[1][4],
                                         const bool (&own)[1], const StepDt<double>& sd,
                                         Acc<double>& acc) {
  double A[4], B[4], um[4], wp[4], wm[4], yE, yEv, L[4], F[4], FR[4], un[4];
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    um[f] = __shfl_up_sync(0xffffffffu, X[0][f], 1);
    B[f] = d64::sub(__shfl_down_sync(0xffffffffu, X[0][f], 1), X[0][f]);
    A[f] = __shfl_up_sync(0xffffffffu, B[f], 1);
  }
  d64::predict1<LIM, SRC>(k, X[0], A, B, sd.dt_2h, sd.dt_2, wp, wm, yE, yEv);
#pragma unroll
  for (int f = 0; f < 4; ++f) L[f] = __shfl_up_sync(0xffffffffu, wp[f], 1);
  hll(k, L, wm, um, X[0], F);
#pragma unroll
  for (int f = 0; f < 4; ++f) FR[f] = __shfl_down_sync(0xffffffffu, F[f], 1);
  if (own[0]) {
    d64::update1<SRC>(X[0], F, FR, yE, yEv, sd.dt, sd.dtdx, un);
    d64::bound<1, SRC>(k, un, acc);
#pragma unroll
    for (int f = 0; f < 4; ++f) X[0][f] = un[f];
  }
}

}  // namespace

}  // namespace sv
