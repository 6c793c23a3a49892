// sv_pairnd.cuh -- the float 2D / 3D MUSCL-Hancock arithmetic (Sec. 2.3:
// eq. 14 reconstruction per axis with xi = 0, the unsplit half-step predictor,
// eq. 13 HLL per axis, eq. 15 update with the source Y, eq. 16 bound) on a
// pair of cells at once in packed f32x2 operations (FFMA2 / FADD2 / FMUL2).
//
// The pair is one thread's cells in two consecutive planes of the marching
// axis (sv_stepnd_pair.cu): component .x the lower plane, .y the upper one.
// Fields are (rho, rho v_1 .. rho v_DIM, E, E_nu), NF = DIM + 3; states are
// f2[NF] (field f of both cells in one register pair).
#pragma once

#include "sv_pair1d.cuh"
#include "sv_reduce.cuh"

namespace sv {
namespace pkn {

using pk::f2;
using pk::add;
using pk::fma;
using pk::mul;
using pk::pair;
using pk::rcp;
using pk::splat;
using pk::sub;

template <int DIM>
struct Prim {
  f2 ir, v[DIM], kin2, p;
};

// Primitive recovery (eq. 5, eq. 7) of two states; PP the pressure policy
// (pk::pressure: 0 float, 2 compensated float).
template <int DIM, int PP>
__device__ __forceinline__ Prim<DIM> prim(const P<float>& k, const f2 (&u)[DIM + 3]) {
  Prim<DIM> q;
  q.ir = rcp(u[0]);
#pragma unroll
  for (int a = 0; a < DIM; ++a) q.v[a] = mul(u[1 + a], q.ir);
  q.kin2 = mul(u[1], q.v[0]);
#pragma unroll
  for (int a = 1; a < DIM; ++a) q.kin2 = fma(u[1 + a], q.v[a], q.kin2);
  q.p = pk::pressure<PP>(k, q.kin2, u[1 + DIM], u[2 + DIM]);
  return q;
}

// div += F(a) - F(b) along axis A (F, G, H of eq. 15; = for the FIRST axis) of
// the states a, b = u +- d/2 with velocities va, vb along A and pressures whose
// difference is dp; (eE, eEv) what v carries of the energies.  No flux is
// formed by itself: the mass fluxes differ by d's momentum, and the other
// fields accumulate v u of both states by fused multiply-adds (13 packed
// operations for the second axis of a 2D pair instead of 20).
template <int DIM, int A, bool FIRST>
__device__ __forceinline__ void add_dflux(const f2 (&d)[DIM + 3], const f2 (&a)[DIM + 3],
                                          const f2 (&b)[DIM + 3], f2 va, f2 vb, f2 dp, f2 aE, f2 aEv,
                                          f2 bE, f2 bEv, f2 (&div)[DIM + 3]) {
  const f2 nvb = mul(vb, splat(-1.0f));
  auto one = [&](f2 x, f2 y, f2& o) { o = fma(va, x, FIRST ? mul(nvb, y) : fma(nvb, y, o)); };
  div[0] = FIRST ? d[1 + A] : add(div[0], d[1 + A]);
#pragma unroll
  for (int c = 0; c < DIM; ++c) one(a[1 + c], b[1 + c], div[1 + c]);
  div[1 + A] = add(div[1 + A], dp);
  one(aE, bE, div[1 + DIM]);
  one(aEv, bEv, div[2 + DIM]);
}

// eq. 13 from the weights wl, wr, wd of the two states' fluxes and of their
// difference: the weights times v once instead of each flux times its weight
// (27 packed operations in 2D instead of 30).  The mass flux keeps the momenta
// themselves, the normal momentum its whole flux (the pressures gathered first
// would round the sum at the size of p twice more: 1000 x 700 cells, 16 steps, error
// against 64 bits 9.35e-8 with the flux, 1.106e-7 so; the same operation count, and
// 8192^2 at 1186 and 1185 us), and the difference its own weight: folding wd into the weights of L and R
// would cancel terms of the size of c u.
template <int DIM, int A>
__device__ __forceinline__ void hll_sum(const f2 (&L)[DIM + 3], const f2 (&R)[DIM + 3], f2 wl, f2 wr,
                                        f2 wd, f2 vl, f2 vr, f2 pl, f2 pr, f2 lE, f2 lEv, f2 rE,
                                        f2 rEv, f2 (&F)[DIM + 3]) {
  const f2 bl = mul(wl, vl), br = mul(wr, vr);
  auto jump = [&](int f) { return sub(L[f], R[f]); };
  F[0] = fma(wd, jump(0), fma(wl, L[1 + A], mul(wr, R[1 + A])));
#pragma unroll
  for (int c = 0; c < DIM; ++c) {
    const f2 s = c == A ? fma(wl, fma(L[1 + c], vl, pl), mul(wr, fma(R[1 + c], vr, pr)))
                        : fma(bl, L[1 + c], mul(br, R[1 + c]));
    F[1 + c] = fma(wd, jump(1 + c), s);
  }
  F[1 + DIM] = fma(wd, jump(1 + DIM), fma(bl, lE, mul(br, rE)));
  F[2 + DIM] = fma(wd, jump(2 + DIM), fma(bl, lEv, mul(br, rEv)));
}

// div += F(u + d/2) - F(u - d/2) along axis A; ok0 / ok1 stay true while both
// extrapolated states of that cell are physical.
template <int DIM, int PP, int A, bool FIRST>
__device__ __forceinline__ void dflux(const P<float>& k, const f2 (&u)[DIM + 3], const f2 (&d)[DIM + 3],
                                      f2 (&div)[DIM + 3], bool& ok0, bool& ok1) {
  constexpr int NF = DIM + 3;
  f2 a[NF], b[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    a[f] = fma(splat(0.5f), d[f], u[f]);
    b[f] = fma(splat(-0.5f), d[f], u[f]);
  }
  const Prim<DIM> pa = prim<DIM, PP>(k, a), pb = prim<DIM, PP>(k, b);
  add_dflux<DIM, A, FIRST>(d, a, b, pa.v[A], pb.v[A], sub(pa.p, pb.p), add(a[1 + DIM], pa.p),
                           a[2 + DIM], add(b[1 + DIM], pb.p), b[2 + DIM], div);
  ok0 = ok0 && fminf(fminf(a[0].x, pa.p.x), fminf(b[0].x, pb.p.x)) > 0.0f;
  ok1 = ok1 && fminf(fminf(a[0].y, pa.p.y), fminf(b[0].y, pb.p.y)) > 0.0f;
}

// Components E and E_nu of Y (eq. 6 closures) of two states.
template <int DIM, int PP, int SRC>
__device__ __forceinline__ void source(const P<float>& k, const f2 (&u)[DIM + 3], f2& yE, f2& yEv) {
  yE = yEv = splat(0.0f);
  if (SRC == 0) return;
  const Prim<DIM> q = prim<DIM, PP>(k, u);
  pk::source<SRC>(k, u[0], mul(q.p, q.ir), u[2 + DIM], yE, yEv);
}

// eq. 13 along axis A at two faces with left states L and right states R; a
// face with a non-physical state uses the cell values, which `cells(fl, fr)`
// supplies (called on that rare path only, so a caller whose cell values sit
// in shared memory loads them only then).  Weights as in pk::hll (all
// non-negative).
template <int DIM, int PP, int A, typename CV>
__device__ __forceinline__ void hll(const P<float>& k, f2 (&L)[DIM + 3], f2 (&R)[DIM + 3],
                                    CV&& cells, f2 (&F)[DIM + 3]) {
  constexpr int NF = DIM + 3;
  Prim<DIM> pl = prim<DIM, PP>(k, L), pr = prim<DIM, PP>(k, R);
  const bool g0 = fminf(fminf(L[0].x, pl.p.x), fminf(R[0].x, pr.p.x)) > 0.0f;
  const bool g1 = fminf(fminf(L[0].y, pl.p.y), fminf(R[0].y, pr.p.y)) > 0.0f;
  if (!(g0 && g1)) {
    f2 fl[NF], fr[NF];
    cells(fl, fr);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      if (!g0) { L[f].x = fl[f].x; R[f].x = fr[f].x; }
      if (!g1) { L[f].y = fl[f].y; R[f].y = fr[f].y; }
    }
    pl = prim<DIM, PP>(k, L);
    pr = prim<DIM, PP>(k, R);
  }
  const f2 gam = splat(k.gamma);
  const f2 cL = pk::sqrt_pos(mul(mul(gam, pl.p), pl.ir));
  const f2 cR = pk::sqrt_pos(mul(mul(gam, pr.p), pr.ir));
  const f2 mL = sub(cL, pl.v[A]), mR = sub(cR, pr.v[A]);
  const f2 qL = add(pl.v[A], cL), qR = add(pr.v[A], cR);
  const f2 nsl = pair(fmaxf(fmaxf(mL.x, mR.x), 0.0f), fmaxf(fmaxf(mL.y, mR.y), 0.0f));
  const f2 sr = pair(fmaxf(fmaxf(qL.x, qR.x), 0.0f), fmaxf(fmaxf(qL.y, qR.y), 0.0f));
  const f2 inv = rcp(add(sr, nsl));
  const f2 wl = mul(sr, inv), wr = mul(nsl, inv), wd = mul(mul(nsl, sr), inv);
  hll_sum<DIM, A>(L, R, wl, wr, wd, pl.v[A], pr.v[A], pl.p, pr.p, add(L[1 + DIM], pl.p), L[2 + DIM],
                  add(R[1 + DIM], pr.p), R[2 + DIM], F);
}

// eq. 16 signal speed and tau key of two updated states, folded for the cells
// whose mask bit is set (bit 0: .x, bit 1: .y).
template <int DIM, int PP, int SRC>
__device__ __forceinline__ void cfl(const P<float>& k, const f2 (&N)[DIM + 3], int mask, float& smax,
                                    float& akey, uint32_t& flags) {
  const Prim<DIM> q = prim<DIM, PP>(k, N);
  const f2 c = pk::sqrt_pos(mul(mul(splat(k.gamma), q.p), q.ir));
  f2 v2 = mul(q.v[0], q.v[0]);
#pragma unroll
  for (int a = 1; a < DIM; ++a) v2 = fma(q.v[a], q.v[a], v2);
  f2 key = splat(-INFINITY);
  if (SRC != 0) key = fma(splat(k.ntau_rho), pk::lg2(N[0]), mul(splat(k.ntau_T), pk::lg2(mul(q.p, q.ir))));
  const float vx = speed_of(v2.x), vy = speed_of(v2.y);
  if (mask & 1) {
    if ((N[0].x > 0.0f) && (q.p.x > 0.0f)) {
      smax = fmaxf(smax, fmaxf(2.0f * vx, __fadd_rn(vx, c.x)));
      if (SRC != 0) akey = fmaxf(akey, key.x);
    } else {
      flags |= FLAG_NONPHYS;
    }
  }
  if (mask & 2) {
    if ((N[0].y > 0.0f) && (q.p.y > 0.0f)) {
      smax = fmaxf(smax, fmaxf(2.0f * vy, __fadd_rn(vy, c.y)));
      if (SRC != 0) akey = fmaxf(akey, key.y);
    } else {
      flags |= FLAG_NONPHYS;
    }
  }
}

}  // namespace pkn
}  // namespace sv
