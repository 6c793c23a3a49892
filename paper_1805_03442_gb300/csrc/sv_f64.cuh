// sv_f64.cuh -- the double-precision arithmetic of one cell (eqs. 5-7, 13-16)
// for 1, 2 and 3 dimensions, written for GB300's narrow FP64 pipe.
//
// The FP64 step kernels are bound by that pipe (two lanes per SM: a warp's
// FP64 instruction holds it 16 cycles, while the integer and float pipes of
// the SM idle), so what counts is the number of FP64 instructions per cell:
//   - a state's recovery forms q = E - E_nu - rho |v|^2 / 2 = p / (gamma - 1)
//     and folds gamma - 1 into the fused multiply-adds that use it;
//   - of the extrapolated states' flux difference the density part is the
//     momentum slope itself;
//   - 1/x is the SFU estimate and one third-order step (three FP64
//     instructions; within 0.507 ulp), sqrt(x) the SFU 1/sqrt estimate and one
//     third-order step (six; 0.531 ulp), over 4 x 10^6 arguments of exponents
//     -300 to 300 and the neighbours of powers of two; minima, maxima, signs and
//     the limiter's decisions are integer instructions on the bit patterns;
//   - the eq. 16 bound is a maximum over all cells: float estimates from the
//     bit patterns decide which cells can hold it, and only those take the
//     square roots and power laws in double.  The maximum found is the one
//     all cells would give, bit for bit (see Bound).
// Every multiply and add is spelled out (no contraction left to the
// compiler), so each kernel built on these functions gives the same bits.
//
// Steps with the paper's tau exponents, minmod, before / after: 1D 10^6 cells
// 597 / 392 us, 2D 500^2 with walls and the medium map 334 / 241 us, 3D
// 150 x 100 x 120 4.71 / 3.74 ms.  Error of a run against 128-bit arithmetic, IEEE square
// roots and two Newton steps per reciprocal / here: 1D spectrum, 10^5 cells, 8
// steps 1.386e-16 / 1.366e-16, 2D wave 300 x 200, 6 steps 1.207e-16 / 1.185e-16.
#pragma once

#include "sv_model.cuh"

namespace sv {
namespace d64 {

__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double fma(double a, double b, double c) { return __fma_rn(a, b, c); }

// The SFU's estimates of 1/x and 1/sqrt(x).
__device__ __forceinline__ double rcp_estimate(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  return y;
}
__device__ __forceinline__ double rsqrt_estimate(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  return y;
}

// 1/x for positive normal x with a normal 1/x: with e = 1 - x y0 of the estimate
// y0 (|e| < 2^-19.9), y0 (1 + e + e^2) has relative error e^3 before rounding.
__device__ __forceinline__ double rcp(double x) {
  const double y = rcp_estimate(x);
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// sqrt(x) for positive normal x: with g = x y0 of the estimate y0 of 1/sqrt(x),
// d = x - g^2 (one rounding) and e = d / x (|e| < 2^-19), sqrt(x) = g (1 - e)^(-1/2) =
// g + d y0 (1/2 + 3 e / 8 + ...).  The binomial series cut there leaves 5 e^3 / 16,
// and d y0^2 = e - e^2 in the place of e another 3 e^3 / 8.
__device__ __forceinline__ double sqrt_pos(double x) {
  const double y = rsqrt_estimate(x);
  const double g = mul(x, y);
  const double t = mul(fma(-g, g, x), y);
  return fma(t, fma(0.375, mul(t, y), 0.5), g);
}

// max(a, b, 0): doubles that are not negative order as their bit patterns do,
// and negative ones lie below zero in both orders.
__device__ __forceinline__ double max0(double a, double b) {
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  const long long m = x > y ? x : y;
  return __longlong_as_double(m > 0 ? m : 0);
}

// The float below a positive double (truncated to 24 bits), from its bits;
// `ok` is cleared outside float's normal range.
__device__ __forceinline__ float trunc_f(double x, bool& ok) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  ok = ok && hi - 0x38100000u < 0x47e00000u - 0x38100000u;
  return __int_as_float((int)(((hi - 0x38000000u) << 3) | (lo >> 29)));
}

// Limited slope from the one-sided differences a, b (LIM 0 minmod, 1 van
// Leer, 2 MC).  Van Leer's quotient is taken only when a b > 0, where a + b is
// normal (a b does not underflow) and carries the sign.
template <int LIM>
__device__ __forceinline__ double limit(double a, double b) {
  if constexpr (LIM == 0) {
    return minmod(a, b);
  } else if constexpr (LIM == 1) {
    const double ab = mul(a, b);
    const double h = mul(ab, rcp(add(a, b)));
    const double d = add(h, h);
    return __double_as_longlong(ab) > 0 ? d : 0.0;
  } else {
    const long long s = (long long)0x8000000000000000ull;
    const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
    if ((ia ^ ib) < 0) return 0.0;
    const long long ma = ia & ~s, mb = ib & ~s;
    const double m = __longlong_as_double(ma < mb ? ma : mb);
    const long long m2 = __double_as_longlong(add(m, m));
    const long long c = __double_as_longlong(mul(0.5, add(a, b))) & ~s;
    return __longlong_as_double((m2 < c ? m2 : c) | (ia & s));
  }
}

// Recovery of a state (eqs. 5, 7): 1/rho, rho |v|^2, q = p / (gamma - 1) and,
// with axis A >= 0, the velocity along it.
struct Prim {
  double ir, v, kin2, q;
};
template <int DIM, int A>
__device__ __forceinline__ Prim prim(const double (&u)[DIM + 3]) {
  Prim r;
  r.ir = rcp(u[0]);
  r.v = A >= 0 ? mul(u[1 + (A < 0 ? 0 : A)], r.ir) : 0.0;
  if (DIM == 1 && A == 0) {
    r.kin2 = mul(u[1], r.v);
  } else {
    double mm = mul(u[1], u[1]);
#pragma unroll
    for (int a = 1; a < DIM; ++a) mm = fma(u[1 + a], u[1 + a], mm);
    r.kin2 = mul(mm, r.ir);
  }
  r.q = fma(-0.5, r.kin2, sub(u[1 + DIM], u[2 + DIM]));
  return r;
}

// x^(n/2) for n >= 1.
__device__ __forceinline__ double half_pow(double x, int n) {
  int i = n >> 1;
  double r = x;
  if (n & 1) r = sqrt_pos(x);
  else --i;
  for (; i > 0; --i) r = mul(r, x);
  return r;
}

// c rho^(kr/2) T^(kT/2) for integers |kr|, |kT| <= 8 with p = rho T: the part
// both powers share is a power of p (the paper's 1/tau ~ rho T^1.5 is
// p sqrt(T)); the negative powers are gathered into one reciprocal.  A whole power
// of T is one for T < 0 too (a half step past p = 0), so it shares whole powers only
// (us per step before / so: 1600 cells 9.34 / 9.33, 10^6 416.3 / 416.2, 2D 500^2
// 233.7 / 233.7, 10^6 with Q and I laws 616 / 622).
__device__ __forceinline__ double law(double c, double rho, double p, double T, int kr, int kT) {
  int kp = 0;
  if (kr > 0 && kT > 0) kp = kr < kT ? kr : kT;
  if (kr < 0 && kT < 0) kp = kr > kT ? kr : kT;
  kp -= (kp % 2) * ((kT & 1) ^ 1);
  kr -= kp;
  kT -= kp;
  double den = 1.0;
  bool any = false;
  auto take = [&](double x, int n) {
    if (n > 0) c = mul(c, half_pow(x, n));
    if (n < 0) {
      const double f = half_pow(x, -n);
      den = any ? mul(den, f) : f;
      any = true;
    }
  };
  take(p, kp);
  take(rho, kr);
  take(T, kT);
  return any ? mul(c, rcp(den)) : c;
}

// Components E and E_nu of Y at a state with recovery r (eq. 6 closures).
template <int SRC>
__device__ __forceinline__ void source(const P<double>& k, double rho, const Prim& r, double Ev,
                                       double& yE, double& yEv) {
  yE = yEv = 0.0;
  if (SRC == 0) return;
  const double p = mul(k.g1, r.q), T = mul(p, r.ir);
  double inv_tau, Q = k.Q0, I = k.Q0;
  if (k.half_tau && (SRC == 1 || k.half_qi)) {
    inv_tau = law(k.inv_tau0, rho, p, T, -k.hk[0], -k.hk[1]);
    if (SRC == 2) {
      Q = law(k.Q0, rho, p, T, k.hk[2], k.hk[3]);
      I = law(k.Q0, rho, p, T, k.hk[4], k.hk[5]);
    }
  } else {
    // other exponents: two logarithms per state, an exponential per closure
    const double lr = log(rho), lT = log(T);
    inv_tau = mul(exp(-fma(k.tau_rho, lr, mul(k.tau_T, lT))), k.inv_tau0);
    if (SRC == 2) {
      Q = mul(k.Q0, exp(fma(k.Q_rho, lr, mul(k.Q_T, lT))));
      I = mul(k.Q0, exp(fma(k.I_rho, lr, mul(k.I_T, lT))));
    }
  }
  if (SRC == 2) yE = mul(rho, sub(Q, I));
  yEv = fma(fma(k.Ck, p, -Ev), inv_tau, mul(rho, Q));
}

// div += F(u + d/2) - F(u - d/2) along axis A (FIRST: div = that); false if
// either state is non-physical.
template <int DIM, int A, bool FIRST>
__device__ __forceinline__ bool dflux(const P<double>& k, const double (&u)[DIM + 3],
                                      const double (&d)[DIM + 3], double (&div)[DIM + 3]) {
  constexpr int NF = DIM + 3;
  double a[NF], b[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    a[f] = fma(0.5, d[f], u[f]);
    b[f] = fma(-0.5, d[f], u[f]);
  }
  const Prim x = prim<DIM, A>(a), y = prim<DIM, A>(b);
  div[0] = FIRST ? d[1 + A] : add(div[0], d[1 + A]);
#pragma unroll
  for (int c = 0; c < DIM; ++c) {
    double s;
    if (DIM == 1) s = x.kin2;
    else s = FIRST ? mul(a[1 + c], x.v) : fma(a[1 + c], x.v, div[1 + c]);
    s = DIM == 1 ? sub(s, y.kin2) : fma(-b[1 + c], y.v, s);
    div[1 + c] = c == A ? fma(k.g1, sub(x.q, y.q), s) : s;
  }
  const double ha = fma(k.g1, x.q, a[1 + DIM]), hb = fma(k.g1, y.q, b[1 + DIM]);
  div[1 + DIM] = fma(-y.v, hb, FIRST ? mul(x.v, ha) : fma(x.v, ha, div[1 + DIM]));
  div[2 + DIM] = fma(-y.v, b[2 + DIM], FIRST ? mul(x.v, a[2 + DIM]) : fma(x.v, a[2 + DIM], div[2 + DIM]));
  return all_positive(a[0], x.q, b[0], y.q);
}

// eq. 13 along axis A; a face with a non-physical state takes the cell values
// that `cells(L, R)` loads (only then).  With -S_L >= 0 every weight is
// non-negative: F = wl F_L + wr F_R + wd (L - R).
template <int DIM, int A, typename CV>
__device__ __forceinline__ void hll(const P<double>& k, double (&L)[DIM + 3], double (&R)[DIM + 3],
                                    CV&& cells, double (&F)[DIM + 3]) {
  Prim x = prim<DIM, A>(L), y = prim<DIM, A>(R);
  if (!all_positive(L[0], x.q, R[0], y.q)) {
    cells(L, R);
    x = prim<DIM, A>(L);
    y = prim<DIM, A>(R);
  }
  const double cL = sqrt_pos(mul(mul(k.gg1, x.q), x.ir));
  const double cR = sqrt_pos(mul(mul(k.gg1, y.q), y.ir));
  const double nsl = max0(sub(cL, x.v), sub(cR, y.v));   // -min(S_L, 0)
  const double sr = max0(add(x.v, cL), add(y.v, cR));    // max(S_R, 0)
  const double inv = rcp(add(sr, nsl));
  const double wl = mul(sr, inv), wr = mul(nsl, inv), wd = mul(wl, nsl);
  auto face = [&](double l, double r, double fl, double fr) {
    return fma(wd, sub(l, r), fma(wl, fl, mul(wr, fr)));
  };
  F[0] = face(L[0], R[0], L[1 + A], R[1 + A]);
#pragma unroll
  for (int c = 0; c < DIM; ++c) {
    double fl, fr;
    if (c == A) {
      fl = DIM == 1 ? fma(k.g1, x.q, x.kin2) : fma(k.g1, x.q, mul(L[1 + c], x.v));
      fr = DIM == 1 ? fma(k.g1, y.q, y.kin2) : fma(k.g1, y.q, mul(R[1 + c], y.v));
    } else {
      fl = mul(L[1 + c], x.v);
      fr = mul(R[1 + c], y.v);
    }
    F[1 + c] = face(L[1 + c], R[1 + c], fl, fr);
  }
  F[1 + DIM] = face(L[1 + DIM], R[1 + DIM], mul(x.v, fma(k.g1, x.q, L[1 + DIM])),
                    mul(y.v, fma(k.g1, y.q, R[1 + DIM])));
  F[2 + DIM] = face(L[2 + DIM], R[2 + DIM], mul(x.v, L[2 + DIM]), mul(y.v, R[2 + DIM]));
}

// The maxima of the eq. 16 bound over the cells a thread has seen, and the
// float thresholds below which a cell cannot change them:
//   s    a float below the largest signal speed found by this thread's block
//        (`share`, a shared-memory word that starts at 0 for every step);
//   l    log2 of the smallest tau / tau0 found by this thread.
// A cell whose estimated speed is below s by more than the estimate's error
// cannot hold the maximum.  A cell's tau matters only if c_tau tau is below
// cfl h / (largest speed), hence below cfl h / s, and below the smallest tau
// found.  Cells that pass either test are evaluated in double, so the block's
// maxima are those of evaluating every cell (a tau that cannot bound dt is
// left out of akey).
struct Bound {
  double smax = 0.0, akey = -INFINITY;
  uint32_t flags = 0;
  float l = INFINITY;
  float* share = nullptr;
};

template <int DIM, int SRC>
__device__ __forceinline__ void bound(const P<double>& k, const double (&u)[DIM + 3], Bound& m) {
  const Prim r = prim<DIM, DIM == 1 ? 0 : -1>(u);
  if (!both_positive(u[0], r.q)) {
    m.flags |= FLAG_NONPHYS;
    return;
  }
  const double c2 = mul(mul(k.gg1, r.q), r.ir);                 // gamma p / rho
  const double v2 = DIM == 1 ? fabs(r.v) : mul(r.kin2, r.ir);   // |v| in 1D, |v|^2 else
  bool ok = true, vok = true;
  const float cf = Ar<float>::sqrt_pos(trunc_f(c2, ok));
  float vf = trunc_f(v2, vok);
  if (DIM > 1) vf = Ar<float>::sqrt_pos(vf);
  // a speed below float's range is at most 1.1e-19; one above it is a fault
  // of the state that the evaluation in double decides on
  if (!vok) {
    vf = 1.1e-19f;
    ok = ok && __double2hiint(v2) < 0x38100000;
  }
  const float s = *(volatile float*)m.share;
  // estimates are within 2^-21 of the values
  const float sf = fmaxf(2.0f * vf, vf + cf) * (1.0f + 0x1p-18f);
  if (!(ok && sf < s)) {
    const double vm = DIM == 1 ? v2 : (v2 > 0x1p-1000 ? sqrt_pos(v2) : 0.0);
    // where it overflows the speed is infinite (dt is then flagged), not inf * 0
    const double c = __double2hiint(c2) < 0x7ff00000 ? sqrt_pos(c2) : c2;
    const double sx = fmax(add(vm, vm), add(vm, c));
    m.smax = fmax(m.smax, sx);
    bool fits = true;
    const float sd = trunc_f(sx, fits);
    if (fits) atomicMax((int*)m.share, __float_as_int(sd));
  }
  if (SRC != 0) {
    bool rok = true;
    const float lr = Ar<float>::lg2(trunc_f(u[0], rok));
    const float lT = Ar<float>::lg2(trunc_f(r.q, rok)) + k.lg_g1 - lr;
    const float lt = fmaf(k.f_tau_rho, lr, k.f_tau_T * lT);      // log2(tau / tau0)
    const float top = fminf(k.l0 - Ar<float>::lg2(*(volatile float*)m.share), m.l);
    // the estimate is within 1e-4 for exponents and logarithms of any state
    // in float's range up to |exponent| 8 and |log2| 10; beyond, always exact
    const float lim = fmaxf(fabsf(lr), fabsf(lT));
    if (!(rok && lim < 10.0f && lt > top + k.l_margin)) {
      const double p = mul(k.g1, r.q), T = mul(p, r.ir);
      double tau;
      if (k.half_tau) tau = law(k.tau0, u[0], p, T, k.hk[0], k.hk[1]);
      else tau = mul(k.tau0, exp(fma(k.tau_rho, log(u[0]), mul(k.tau_T, log(T)))));
      m.akey = fmax(m.akey, -tau);
      if (rok && lim < 10.0f) m.l = fminf(m.l, lt);
    }
  }
}

// Slopes d from the one-sided differences A (left) and B (right), the
// positivity guard, the half-step predictor, the + and - face states and the
// half-step source of one 1D cell.
template <int LIM, int SRC>
__device__ __forceinline__ void predict1(const P<double>& k, const double (&u)[4],
                                         const double (&A)[4], const double (&B)[4], double dt_2h,
                                         double dt_2, double (&wp)[4], double (&wm)[4], double& yEh,
                                         double& yEvh) {
  double d[4], div[4];
#pragma unroll
  for (int f = 0; f < 4; ++f) d[f] = limit<LIM>(A[f], B[f]);
  if (!dflux<1, 0, true>(k, u, d, div)) {
#pragma unroll
    for (int f = 0; f < 4; ++f) d[f] = div[f] = 0.0;
  }
  double uh[4];
#pragma unroll
  for (int f = 0; f < 4; ++f) uh[f] = fma(-dt_2h, div[f], u[f]);
  if (SRC != 0) {
    double yE, yEv;
    source<SRC>(k, u[0], prim<1, -1>(u), u[3], yE, yEv);
    if (SRC == 2) uh[2] = fma(dt_2, yE, uh[2]);
    uh[3] = fma(dt_2, yEv, uh[3]);
  }
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    wp[f] = fma(0.5, d[f], uh[f]);
    wm[f] = fma(-0.5, d[f], uh[f]);
  }
  yEh = yEvh = 0.0;
  if (SRC != 0) source<SRC>(k, uh[0], prim<1, -1>(uh), uh[3], yEh, yEvh);
}

// Heun stages: guarded face states at the stage's own time level and Y(u).
template <int LIM, int SRC>
__device__ __forceinline__ void level1(const P<double>& k, const double (&u)[4],
                                       const double (&A)[4], const double (&B)[4],
                                       double (&wp)[4], double (&wm)[4], double& yE, double& yEv) {
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const double d = limit<LIM>(A[f], B[f]);
    wp[f] = fma(0.5, d, u[f]);
    wm[f] = fma(-0.5, d, u[f]);
  }
  const Prim x = prim<1, -1>(wp), y = prim<1, -1>(wm);
  if (!all_positive(wp[0], x.q, wm[0], y.q)) {
#pragma unroll
    for (int f = 0; f < 4; ++f) wp[f] = wm[f] = u[f];
  }
  yE = yEv = 0.0;
  if (SRC != 0) source<SRC>(k, u[0], prim<1, -1>(u), u[3], yE, yEv);
}

// Conservative update (eq. 15) of a 1D cell.
template <int SRC>
__device__ __forceinline__ void update1(const double (&u)[4], const double (&Fl)[4],
                                        const double (&Fr)[4], double yE, double yEv, double dt,
                                        double dtdx, double (&un)[4]) {
#pragma unroll
  for (int f = 0; f < 4; ++f) un[f] = fma(-dtdx, sub(Fr[f], Fl[f]), u[f]);
  if (SRC == 2) un[2] = fma(dt, yE, un[2]);
  if (SRC != 0) un[3] = fma(dt, yEv, un[3]);
}

}  // namespace d64
}  // namespace sv
