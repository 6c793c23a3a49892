// sv_stepnd.cu -- fused 2D / 3D unsplit MUSCL-Hancock steps in double (Sec. 2.3:
// eq. 15 with both flux differences F and G -- and the analogous z flux in
// 3D -- in one update; eq. 14 face states per axis with xi = 0; eq. 13 HLL per
// axis; source Y at the half step; eq. 16 reduction), and the dispatch of the
// float steps to their kernels.  Bound by the FP64 pipe: the arithmetic is that
// of sv_f64.cuh.
//
// Work decomposition ("marching planes").  Each block owns a transverse tile
// (TX threads along x in 2D; TX x TY threads over x-y in 3D) and a segment of
// planes along the outermost axis (y in 2D, z in 3D).  Thread (tx, ty) owns
// the column of cells at one transverse position; the outer ring of threads is
// a one-cell halo whose predictors feed the tile's faces but which update
// nothing.  Per plane q the block
//   a. publishes plane q's states in shared memory (the halo threads also load
//      the second ring, needed by their slopes),
//   b. computes slopes (all axes; the marching-axis slope from the planes
//      q-1, q, q+1 held in registers), the positivity guard and the half-step
//      predictor of plane q -- once per cell,
//   c. publishes the +face states of the transverse axes and computes each
//      cell's left transverse faces (HLL, once per face),
//   d. publishes those fluxes and forms the transverse flux divergence,
//   e. computes the marching-axis face between planes q-1 and q,
//   f. updates plane q-1 (all its faces are now known) and folds its
//      signal speed / tau bound for the next dt.
// Three barriers per plane.  The warm-up plane before the segment and the
// plane beyond it skip the transverse faces, which nothing uses there (500^2
// with walls, 7-row segments: 261 -> 241 us per step; 64^3: 587 -> 546).
// Each thread streams its own column (and the halo
// threads their second-ring cells) through a per-thread ring of kPlaneRing
// planes in shared memory with cp.async, four planes ahead of the one being
// computed; copies are coalesced along x.
#include "sv_internal.h"
#include "sv_ndbnd.cuh"
#include "sv_step1d.cuh"      // cp.async helpers

namespace sv {

// Planes per thread ring (a power of two; four planes are in flight).
constexpr int kPlaneRing = 8;

// Slots of the second-ring cells: two per tile row (x ring) and, in 3D, two
// per tile column (y ring).
template <int DIM, int TX, int TY> struct HaloSlots {
  static constexpr int N = 2 * TY + (DIM == 3 ? 2 * TX : 0);
};

template <typename R, int DIM, int TX, int TY>
constexpr size_t stepnd_smem() {
  constexpr int NF = DIM + 3, SY = DIM == 3 ? TY + 2 : 1, NT = TX * TY;
  return sizeof(R) * ((size_t)NF * SY * (TX + 2) + 2 * (size_t)(DIM - 1) * NF * TY * TX +
                      (size_t)kPlaneRing * NF * NT + (size_t)kPlaneRing * NF * HaloSlots<DIM, TX, TY>::N);
}

// DIM 2: TY must be 1; marching axis y.  DIM 3: marching axis z.
// BND: a 2D grid with walls or outflow on some side, or a medium map / driven
// cells; without it every axis is periodic (the compiled-out general path
// costs the periodic kernel 8%).
template <int LIM, int SRC, int DIM, int TX, int TY, int MINB, bool BND>
__global__ void __launch_bounds__(TX * TY, MINB)
stepnd_kernel(const KParams kp, double* __restrict__ bufA, double* __restrict__ bufB,
              Ctl* __restrict__ ctl, int64_t nx, int64_t ny, int64_t nz, int tiles_x, int tiles_y,
              int nseg) {
  using R = double;
  constexpr int NF = DIM + 3;
  constexpr int NT = TX * TY;
  constexpr int SY = DIM == 3 ? TY + 2 : 1;     // rows of the shared state plane
  constexpr int AM = DIM - 1;                   // marching axis
  // dynamic shared memory: sU[NF][SY][TX+2], sW[DIM-1][NF][TY][TX],
  // sF[DIM-1][NF][TY][TX], sR[D][NF][NT] (own-column ring), sH[D][NF][NH]
  // (second-ring cells of the halo threads)
  constexpr int D = kPlaneRing, NH = HaloSlots<DIM, TX, TY>::N;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  R (*sU)[SY][TX + 2] = reinterpret_cast<R (*)[SY][TX + 2]>(smem_raw);
  R (*sW)[NF][TY][TX] = reinterpret_cast<R (*)[NF][TY][TX]>(smem_raw + sizeof(R) * NF * SY * (TX + 2));
  R (*sF)[NF][TY][TX] = reinterpret_cast<R (*)[NF][TY][TX]>(
      smem_raw + sizeof(R) * (NF * SY * (TX + 2) + (DIM - 1) * NF * TY * TX));
  R (*sR)[NF][NT] = reinterpret_cast<R (*)[NF][NT]>(
      smem_raw + sizeof(R) * (NF * SY * (TX + 2) + 2 * (DIM - 1) * NF * TY * TX));
  R (*sH)[NF][NH] = reinterpret_cast<R (*)[NF][NH]>(
      smem_raw + sizeof(R) * (NF * SY * (TX + 2) + 2 * (DIM - 1) * NF * TY * TX + D * NF * NT));

  const StepCtl sc = block_step_ctl(ctl);
  if (!(sc.dt > 0.0)) return;
  const R* __restrict__ Uin = sc.cur ? bufB : bufA;
  R* __restrict__ Uout = sc.cur ? bufA : bufB;
  const P<R> k(kp);
  const StepDt<R> sd(sc);
  const R dt = sd.dt, dtdx = sd.dtdx, dt_2h = sd.dt_2h, dt_2 = sd.dt_2;

  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
  const int seg = blockIdx.x % nseg;
  const int tile = blockIdx.x / nseg;
  const int tile_x = tile % tiles_x, tile_y = tile / tiles_x;
  // Cell and field offsets in 32 bits: the launch admits grids whose fields
  // hold fewer than 2^31 values in all (stepnd_launch).
  using I = int;
  const I gx = (I)tile_x * (TX - 2) - 1 + tx;
  const I gy = DIM == 3 ? (I)tile_y * (TY - 2) - 1 + ty : 0;
  const I M = (I)(DIM == 3 ? nz : ny);                      // planes
  const I plane = (I)(DIM == 3 ? nx * ny : nx);             // cells per plane
  const I ncell = plane * M;
  const I q0 = (I)((int64_t)seg * M / nseg), q1 = (I)((int64_t)(seg + 1) * M / nseg);
  const I nxi = (I)nx, nyi = (I)ny;
  const bool interior = tx >= 1 && tx <= TX - 2 && gx < nxi &&
                        (DIM == 2 || (ty >= 1 && ty <= TY - 2 && gy < nyi));
  // 2D boundaries: x sides kp.bc_lo / bc_hi, y sides (the marching axis)
  // kp.bc_ylo / bc_yhi; 3D is periodic.  Ghost positions load the mapped cell;
  // the reversed momenta of wall ghosts are applied when the planes are read.
  static_assert(!BND || DIM == 2, "boundaries and media are 2D only");
  bool fx_own = false, fx_rx = false;
  const I wx = BND ? map_axis(gx, nxi, kp.bc_lo, kp.bc_hi, fx_own) : wrap(gx, nxi);
  const I wy = DIM == 3 ? wrap(gy, nyi) : 0;
  const I col = DIM == 3 ? wy * nxi + wx : wx;               // index within a plane
  // second-ring positions loaded by the halo threads
  const bool ringx = (tx == 0) || (tx == TX - 1);
  const I col_rx = (DIM == 3 ? wy * nxi : 0) +
                   (BND ? map_axis(gx + (tx == 0 ? -1 : 1), nxi, kp.bc_lo, kp.bc_hi, fx_rx)
                        : wrap(gx + (tx == 0 ? -1 : 1), nxi));
  // plane of the marching axis holding position p, and whether it is a wall ghost
  auto plane_of = [&](I p, bool& fy) -> I {
    if (!BND) {
      fy = false;
      return wrap(p, M);
    }
    return map_axis(p, M, kp.bc_ylo, kp.bc_yhi, fy);
  };
  const bool medium = BND && kp.act_lo != nullptr;
  const bool pulses = BND && kp.pul_lo != nullptr;
  const bool ringy = DIM == 3 && ((ty == 0) || (ty == TY - 1));
  const I col_ry = DIM == 3 ? wrap(gy + (ty == 0 ? -1 : 1), nyi) * nxi + wx : 0;
  const int oy = DIM == 3 ? ty + 1 : 0;

  Acc<R> acc(bound_word());

  const int tid = threadIdx.x;
  const int hx = ty * 2 + (tx == 0 ? 0 : 1);                              // x-ring slot
  const int hy = 2 * TY + tx * 2 + (ty == 0 ? 0 : 1);                     // y-ring slot
  // copy plane p of the own column (p <= q1 + 1) and of the second ring
  // (p <= q1) into ring slot p mod D; always commit a group
  auto issue = [&](I p) {
    const int sl = (int)(p & (D - 1));
    if (p <= q1 + 1) {
      bool fy;
      const I o = plane_of(p, fy) * plane;
#pragma unroll
      for (int f = 0; f < NF; ++f) cp_async<sizeof(R)>(&sR[sl][f][tid], Uin + f * ncell + o + col);
      if (p <= q1) {
        if (ringx)
#pragma unroll
          for (int f = 0; f < NF; ++f) cp_async<sizeof(R)>(&sH[sl][f][hx], Uin + f * ncell + o + col_rx);
        if (ringy)
#pragma unroll
          for (int f = 0; f < NF; ++f) cp_async<sizeof(R)>(&sH[sl][f][hy], Uin + f * ncell + o + col_ry);
      }
    }
    cp_async_commit();
  };

  R Um1[NF], Uq[NF], Up1[NF];
  R Wm_prev[NF], D_prev[NF], H_prev[NF], yE_prev = 0, yEv_prev = 0;
#pragma unroll
  for (int f = 0; f < NF; ++f) Wm_prev[f] = D_prev[f] = H_prev[f] = (R)0;
  auto pidx = [&](I q) {
    bool fy;
    return plane_of(q, fy) * plane;
  };
  for (I p = q0 - 2; p <= q0 + D - 4; ++p) issue(p);    // D - 1 planes ahead

  for (I q = q0 - 1; q <= q1; ++q) {
    // a. planes q-1, q, q+1 of the own column and plane q's second ring have
    //    landed; publish plane q
    cp_async_wait<D - 4>();
    const int sm = (int)((q - 1) & (D - 1)), s0 = (int)(q & (D - 1)), sp = (int)((q + 1) & (D - 1));
    bool fym, fy0, fyp;
    const I jq = plane_of(q, fy0);
    plane_of(q - 1, fym);
    plane_of(q + 1, fyp);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      Um1[f] = sR[sm][f][tid];
      Uq[f] = sR[s0][f][tid];
      Up1[f] = sR[sp][f][tid];
    }
    if (BND) {
      if (fx_own) {
        Um1[1] = -Um1[1];
        Uq[1] = -Uq[1];
        Up1[1] = -Up1[1];
      }
      if (fym) Um1[2] = -Um1[2];
      if (fy0) Uq[2] = -Uq[2];
      if (fyp) Up1[2] = -Up1[2];
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      sU[f][oy][tx + 1] = Uq[f];
      if (ringx) {
        R v = sH[s0][f][hx];
        if (BND && ((f == 1 && fx_rx) || (f == 2 && fy0))) v = -v;
        sU[f][oy][tx == 0 ? 0 : TX + 1] = v;
      }
      if (DIM == 3 && ringy) sU[f][ty == 0 ? 0 : SY - 1][tx + 1] = sH[s0][f][hy];
    }
    // medium of this cell (the mapped cell of a ghost): active or frozen
    const bool active = !medium || (wx >= __ldg(kp.act_lo + jq) && wx < __ldg(kp.act_hi + jq));
    issue(q + D - 2);    // reuses the slot of plane q-2 (read one barrier ago)
    __syncthreads();

    // b. slopes and predictor of plane q
    R d[DIM][NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      d[0][f] = d64::limit<LIM>(d64::sub(Uq[f], sU[f][oy][tx]), d64::sub(sU[f][oy][tx + 2], Uq[f]));
      if (DIM == 3)
        d[1][f] = d64::limit<LIM>(d64::sub(Uq[f], sU[f][oy - 1][tx + 1]),
                                  d64::sub(sU[f][oy + 1][tx + 1], Uq[f]));
      d[AM][f] = d64::limit<LIM>(d64::sub(Uq[f], Um1[f]), d64::sub(Up1[f], Uq[f]));
    }
    R div[NF];
    bool ok = d64::dflux<DIM, 0, true>(k, Uq, d[0], div);
    ok = d64::dflux<DIM, 1, false>(k, Uq, d[1], div) && ok;
    if (DIM == 3) ok = d64::dflux<DIM, DIM - 1, false>(k, Uq, d[AM], div) && ok;
    if (!ok) {
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        div[f] = 0.0;
#pragma unroll
        for (int a = 0; a < DIM; ++a) d[a][f] = 0.0;
      }
    }
    R uh[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) uh[f] = d64::fma(-dt_2h, div[f], Uq[f]);
    R yEh = 0.0, yEvh = 0.0;
    if (SRC != 0 && active) {         // a frozen cell has no source
      R yE, yEv;
      d64::source<SRC>(k, Uq[0], d64::prim<DIM, -1>(Uq), Uq[2 + DIM], yE, yEv);
      if (SRC == 2) uh[1 + DIM] = d64::fma(dt_2, yE, uh[1 + DIM]);
      uh[2 + DIM] = d64::fma(dt_2, yEv, uh[2 + DIM]);
      d64::source<SRC>(k, uh[0], d64::prim<DIM, -1>(uh), uh[2 + DIM], yEh, yEvh);
    }

    R Dq[NF];
    if (q < q0 || q == q1) {
      // a warm-up plane (only its marching + states are used) or the plane
      // beyond the segment (only its marching - states): no transverse faces
#pragma unroll
      for (int f = 0; f < NF; ++f) Dq[f] = 0.0;
      __syncthreads();               // plane q has been read before the next is published
    } else {
    // c. transverse faces: publish +states, take the left neighbour's
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      sW[0][f][ty][tx] = d64::fma(0.5, d[0][f], uh[f]);
      if (DIM == 3) sW[DIM == 3 ? 1 : 0][f][ty][tx] = d64::fma(0.5, d[1][f], uh[f]);
    }
    __syncthreads();
    R Fx[NF], Fy[NF];
    {
      R l[NF], r[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        l[f] = sW[0][f][ty][tx > 0 ? tx - 1 : tx];
        r[f] = d64::fma(-0.5, d[0][f], uh[f]);
      }
      d64::hll<DIM, 0>(k, l, r,
                       [&](R (&L)[NF], R (&Rr)[NF]) {
#pragma unroll
                         for (int f = 0; f < NF; ++f) {
                           L[f] = sU[f][oy][tx];
                           Rr[f] = Uq[f];
                         }
                       },
                       Fx);
      if (DIM == 3) {
#pragma unroll
        for (int f = 0; f < NF; ++f) {
          l[f] = sW[DIM == 3 ? 1 : 0][f][ty > 0 ? ty - 1 : ty][tx];
          r[f] = d64::fma(-0.5, d[1][f], uh[f]);
        }
        d64::hll<DIM, 1>(k, l, r,
                         [&](R (&L)[NF], R (&Rr)[NF]) {
#pragma unroll
                           for (int f = 0; f < NF; ++f) {
                             L[f] = sU[f][oy > 0 ? oy - 1 : oy][tx + 1];
                             Rr[f] = Uq[f];
                           }
                         },
                         Fy);
      }
    }
    // d. transverse flux divergence of plane q
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      sF[0][f][ty][tx] = Fx[f];
      if (DIM == 3) sF[DIM == 3 ? 1 : 0][f][ty][tx] = Fy[f];
    }
    __syncthreads();
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      Dq[f] = d64::sub(sF[0][f][ty][tx < TX - 1 ? tx + 1 : tx], Fx[f]);
      if (DIM == 3)
        Dq[f] = d64::add(Dq[f], d64::sub(sF[DIM == 3 ? 1 : 0][f][ty < TY - 1 ? ty + 1 : ty][tx], Fy[f]));
    }

    }

    // e. marching-axis face between planes q-1 and q
    R Hq[NF];
    if (q >= q0) {
      R Wm[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f) Wm[f] = d64::fma(-0.5, d[AM][f], uh[f]);
      d64::hll<DIM, AM>(k, Wm_prev, Wm,
                        [&](R (&L)[NF], R (&Rr)[NF]) {
#pragma unroll
                          for (int f = 0; f < NF; ++f) {
                            L[f] = Um1[f];
                            Rr[f] = Uq[f];
                          }
                        },
                        Hq);
    }

    // f. update of plane q-1
    if (q > q0 && interior) {
      R un[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f)
        un[f] = d64::fma(-dtdx, d64::sub(d64::add(D_prev[f], Hq[f]), H_prev[f]), Um1[f]);
      if (SRC == 2) un[1 + DIM] = d64::fma(dt, yE_prev, un[1 + DIM]);
      if (SRC != 0) un[2 + DIM] = d64::fma(dt, yEv_prev, un[2 + DIM]);
      // a driven cell holds the pulsating source at the new time level
      if (pulses && gx >= __ldg(kp.pul_lo + (q - 1)) && gx < __ldg(kp.pul_hi + (q - 1)))
        pulse_state<R, NF>(kp, sc.t + sc.dt, un);
      const I o = pidx(q - 1) + col;
#pragma unroll
      for (int f = 0; f < NF; ++f) Uout[f * ncell + o] = un[f];
      d64::bound<DIM, SRC>(k, un, acc);
    }

    // rotate the plane window
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      Wm_prev[f] = d64::fma(0.5, d[AM][f], uh[f]);
      D_prev[f] = Dq[f];
      H_prev[f] = Hq[f];
    }
    yE_prev = yEh;
    yEv_prev = yEvh;
  }
  cp_async_wait<0>();
  reduce_and_finalize<R, NT>(ctl, kp, acc.smax, acc.akey, acc.flags, true);
}

// ------------------------------------------------------------------ launch

template <int DIM> struct Cfg;
template <> struct Cfg<2> { static constexpr int TX = 128, TY = 1, MINB = 2, SEG = 256; };
template <> struct Cfg<3> { static constexpr int TX = 16, TY = 16, MINB = 1, SEG = 128; };

// With `n` null only the kernel's shared-memory attribute is set (done once per
// solver at init, outside any stream capture).  `nseg` = segments of the
// marching axis (march_segments).
template <int LIM, int SRC, int DIM>
static cudaError_t launch_nd(const KParams& kp, void* a, void* b, Ctl* ctl, const int64_t* n,
                            int nseg, cudaStream_t st) {
  using G = Cfg<DIM>;
  constexpr size_t smem = stepnd_smem<double, DIM, G::TX, G::TY>();
  const bool bnd = DIM == 2 && (kp.bc_lo != BC_PERIODIC || kp.bc_hi != BC_PERIODIC ||
                                kp.bc_ylo != BC_PERIODIC || kp.bc_yhi != BC_PERIODIC ||
                                kp.act_lo != nullptr || kp.pul_lo != nullptr);
  auto fn = bnd ? stepnd_kernel<LIM, SRC, DIM, G::TX, G::TY, G::MINB, DIM == 2>
                : stepnd_kernel<LIM, SRC, DIM, G::TX, G::TY, G::MINB, false>;
  if (!n) {
    cudaError_t e = cudaFuncSetAttribute(stepnd_kernel<LIM, SRC, DIM, G::TX, G::TY, G::MINB, false>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess || DIM != 2) return e;
    return cudaFuncSetAttribute(stepnd_kernel<LIM, SRC, DIM, G::TX, G::TY, G::MINB, DIM == 2>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  }
  const int64_t nx = n[0], ny = n[1], nz = DIM == 3 ? n[2] : 1;
  const int tiles_x = (int)((nx + G::TX - 3) / (G::TX - 2));
  const int tiles_y = DIM == 3 ? (int)((ny + G::TY - 3) / (G::TY - 2)) : 1;
  if (nseg < 1 || nseg > (DIM == 3 ? nz : ny)) return cudaErrorInvalidValue;
  const int64_t blocks = (int64_t)tiles_x * tiles_y * nseg;
  if (blocks > 0x7fffffff) return cudaErrorInvalidConfiguration;
  fn<<<(int)blocks, G::TX * G::TY, smem, st>>>(kp, (double*)a, (double*)b, ctl, nx, ny, nz, tiles_x, tiles_y,
                                               nseg);
  return cudaGetLastError();
}

template <int LIM, int SRC, int DIM>
static cudaError_t by_prec(int precision, const KParams& kp, void* a, void* b, Ctl* ctl,
                           const int64_t* n, int nseg, cudaStream_t st) {
  switch (precision) {
    case PREC_FP64: return launch_nd<LIM, SRC, DIM>(kp, a, b, ctl, n, nseg, st);
    default:
      // the float policies: in 2D packed plane pairs
      // (sv_stepnd_pair.cu); in 3D each cell's fields in packed pairs
      // (sv_stepnd3f.cu: plane pairs need 242 registers there, one block per
      // SM, and ran 17% slower than one cell per thread)
      if constexpr (DIM == 2) return stepnd_pair_launch(DIM, precision, kp, a, b, ctl, n, nseg, st);
      else return stepnd3f_launch(precision, kp, a, b, ctl, n, nseg, st);
  }
}

template <int LIM, int DIM>
static cudaError_t by_src(int precision, const KParams& kp, void* a, void* b, Ctl* ctl,
                          const int64_t* n, int nseg, cudaStream_t st) {
  if (kp.frozen) return by_prec<LIM, 0, DIM>(precision, kp, a, b, ctl, n, nseg, st);
  if (kp.qi_zero) return by_prec<LIM, 1, DIM>(precision, kp, a, b, ctl, n, nseg, st);
  return by_prec<LIM, 2, DIM>(precision, kp, a, b, ctl, n, nseg, st);
}

template <int DIM>
static cudaError_t by_lim(int precision, const KParams& kp, void* a, void* b, Ctl* ctl,
                          const int64_t* n, int nseg, cudaStream_t st) {
  switch (kp.limiter) {
    case 1: return by_src<1, DIM>(precision, kp, a, b, ctl, n, nseg, st);
    case 2: return by_src<2, DIM>(precision, kp, a, b, ctl, n, nseg, st);
    default: return by_src<0, DIM>(precision, kp, a, b, ctl, n, nseg, st);
  }
}

// Two 2D blocks on an SM take 1.75 times one block's iteration (28.4 and 16.2
// us); the two extra iterations skip the transverse faces and so cost 1.2.
template <int DIM>
static MarchShape shape_of() {
  using G = Cfg<DIM>;
  return {G::TX - 2, DIM == 3 ? G::TY - 2 : 0, 1, 1.2, G::MINB, {1.0, 1.75, 0.0}, G::SEG};
}

MarchShape stepnd_shape(int dim, int precision) {
  if (precision == PREC_FP64) return dim == 2 ? shape_of<2>() : shape_of<3>();
  return dim == 2 ? stepnd_pair_shape() : stepnd3f_shape();
}

int stepnd_grid(int dim, int precision, const KParams& kp) {
  cudaError_t e = cudaErrorInvalidValue;
  if (dim == 2) e = by_lim<2>(precision, kp, nullptr, nullptr, nullptr, nullptr, 0, nullptr);
  if (dim == 3) e = by_lim<3>(precision, kp, nullptr, nullptr, nullptr, nullptr, 0, nullptr);
  return e == cudaSuccess ? 1 : 0;
}

cudaError_t stepnd_launch(int dim, int precision, const KParams& kp, void* a, void* b, Ctl* ctl,
                          const int64_t* n, int nseg, cudaStream_t st) {
  if (!n) return cudaErrorInvalidValue;
  int64_t ncell = n[0] * n[1] * (dim == 3 ? n[2] : 1);
  if (ncell * (dim + 3) >= (1LL << 31)) return cudaErrorInvalidValue;
  if (dim == 2) return by_lim<2>(precision, kp, a, b, ctl, n, nseg, st);
  if (dim == 3) return by_lim<3>(precision, kp, a, b, ctl, n, nseg, st);
  return cudaErrorInvalidValue;
}

}  // namespace sv
