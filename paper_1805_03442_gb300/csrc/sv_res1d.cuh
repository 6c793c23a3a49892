// sv_res1d.cuh -- many 1D MUSCL-Hancock steps (Sec. 2.3: eqs. 13-15 with
// xi = 0, source Y, eq. 16 reduction) in one launch with the state held in
// registers: grids of up to one block per SM.
//
// A step of such a grid is a chain of latencies, so this kernel leaves nothing
// in the chain but the arithmetic and one exchange:
//   - a warp owns a run of at most OWN consecutive cells for the whole launch
//     (60 in float, two cells per lane in packed pairs; 28 in double, one per
//     lane), plus two halo cells on either side whose faces it computes
//     itself, so that within a step lanes exchange only shuffles;
//   - after the update each warp publishes its first and last two cells and
//     its dt bounds: to the block's other warps through shared memory, to the
//     other blocks through words of 8 bytes holding a tag and 4 bytes of data
//     (an 8-byte store is seen whole, so a word with the step's tag is valid by
//     itself: no fence, no counter, no atomic);
//   - every block receives the bounds of all blocks in a mailbox of its own and
//     computes the next dt itself, with the arithmetic of the per-step finalize.
// One block: one barrier per step.  Several: two barriers and one trip through
// L2.  Per cell the arithmetic is that of the step kernels, function for
// function, so the states are bitwise those of per-step launches.
//
// Words alternate between two sets by step parity.  A block writes step s + 2's
// words after it has seen every block's step s + 1, which each published after
// it had read all of step s: nothing unread is overwritten.  At the start of a
// launch each block clears its own words; tags carry the launch's number (the
// control block's generation, which each launch that steps and each upload
// advances), so those of the launch before are not taken for this one's, nor in
// the replays of a captured launch.
//
// Measured, us per step, per-step launches / here: float 200 cells 7.6 / 1.6,
// 1000 7.7 / 2.2, 10^4 6.0 / 3.0, 10^5 7.3 / 3.9, 1.8 x 10^5 6.5 / 4.7; double
// 1600 48 / 9.5, 3 x 10^4 49 / 18.  What is left is the chain of one warp's step
// (1.6 us in float) and the exchange (0.6 us between 5 blocks, 1.3 us between
// 152).  With one mailbox that all blocks poll instead of one each, the 152
// blocks of 10^5 cells took 6.4 us: every SM read the same 19 lines.
//
// Every wait is bounded in time and polls: a block that gives up raises
// FLAG_STALL and leaves, and the others' waits then run out likewise.
#pragma once

#include "sv_internal.h"
#include "sv_window1d.cuh"

namespace sv {

namespace {

constexpr uint64_t kResStallNs = 2000000000ull;   // give up a wait after 2 s
constexpr uint32_t kResStallIters = 1u << 24;      // ... or after this many polls

template <typename R> struct ResWarps;
template <> struct ResWarps<float> { static constexpr int N = kResWarpsF; };
template <> struct ResWarps<double> { static constexpr int N = kResWarpsD; };

__device__ __forceinline__ void put_word(uint64_t* p, uint32_t tag, uint32_t v) {
  const uint64_t w = ((uint64_t)tag << 32) | v;
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ uint64_t get_word(const uint64_t* p) {
  uint64_t w;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  return w;
}
__device__ __forceinline__ uint64_t res_timer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void put_words2(uint64_t* p, uint32_t tag, uint32_t v0, uint32_t v1) {
  const uint64_t a = ((uint64_t)tag << 32) | v0, b = ((uint64_t)tag << 32) | v1;
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void get_words2(const uint64_t* p, uint64_t& a, uint64_t& b) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}

// Wait until the NV words at p (NV 1, or even: 16-byte aligned) carry `tag`
// (whose bit 0 is data); lanes without `need` return at once.  False when the
// limits run out.
template <int NV>
__device__ __forceinline__ bool wait_words(const uint64_t* p, bool need, uint32_t tag,
                                           uint64_t (&w)[NV], int polls) {
  const uint32_t limit = polls > 0 ? (uint32_t)polls : kResStallIters;
  uint64_t t0 = 0;
  for (uint32_t it = 0; it < limit; ++it) {
    bool ok = true;
    if (need) {
      if constexpr (NV == 1) {
        w[0] = get_word(p);
      } else {
#pragma unroll
        for (int n = 0; n < NV; n += 2) get_words2(p + n, w[n], w[n + 1]);
      }
#pragma unroll
      for (int n = 0; n < NV; ++n) ok = ok && ((uint32_t)(w[n] >> 32) | 1u) == (tag | 1u);
    }
    if (ok) return true;
    if ((it & 1023u) == 1023u) {
      const uint64_t t = res_timer();
      if (!t0) t0 = t;
      else if (t - t0 > kResStallNs) return false;
    }
  }
  return false;
}

__device__ __forceinline__ uint32_t word_of(float x, int) { return __float_as_uint(x); }
__device__ __forceinline__ uint32_t word_of(double x, int i) {
  return i ? (uint32_t)__double2hiint(x) : (uint32_t)__double2loint(x);
}
__device__ __forceinline__ void from_words(const uint32_t* w, float& x) { x = __uint_as_float(w[0]); }
__device__ __forceinline__ void from_words(const uint32_t* w, double& x) {
  x = __hiloint2double((int)w[1], (int)w[0]);
}

template <typename R, int MAXW>
struct ResSmem {
  R edge[2][MAXW][2][2][4];        // by parity: each warp's first / last two cells
  R smax[2][MAXW], akey[2][MAXW];
  uint32_t fl[2][MAXW];
  uint32_t halo[2][2][4][sizeof(R) / 4];   // the neighbour blocks' cells: side, cell, field
  double t;                        // the run's time, near t_end
  R bmax[kResBlocks / 32], bkey[kResBlocks / 32];   // maxima over 32 blocks each
  uint32_t bflags[kResBlocks / 32];
  float word[2];                   // speed threshold of the double bound, by parity
  int stall;
};

// Up to nmax steps; stops once the next dt is 0 (t_end reached or a flag
// raised).  `words`: ResWords of the exchange (several blocks only); `wtot`:
// warps that own cells.
template <typename R, int PP, int LIM, int SRC>
__global__ void __launch_bounds__(ResWarps<R>::N * 32, 1)
res1d_kernel(const KParams kp, R* bufA, R* bufB, Ctl* ctl, uint64_t* words, int N, int wtot,
             int nmax) {
  constexpr int CPL = Win<R>::CPL, MAXW = ResWarps<R>::N, NW = sizeof(R) / 4;
  __shared__ ResSmem<R, MAXW> S;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int W = blockDim.x >> 5, G = gridDim.x, b = blockIdx.x;
  const int gw = b * W + w;
  const int lw = min(W, wtot - b * W) - 1;      // the block's last warp with cells
  const bool live = w <= lw;

  if (threadIdx.x == 0) {
    S.word[0] = S.word[1] = 0.0f;
    // read by one thread: a block that has started already may raise it meanwhile,
    // and all threads of this one have to leave or stay together
    S.stall = (vload(&ctl->flags) & FLAG_STALL) != 0;
  }
  // words by parity: block i's mailbox has NM bounds from each block (a private
  // one: polled by block i alone, so that no line is read by every SM), and
  // its edges are the first and last two cells
  constexpr int NM = 2 * NW, NE = 8 * NW;
  uint64_t* const mw = words;                             // [2][G][G][NM]
  uint64_t* const ew = words + (size_t)2 * G * G * NM;    // [2][G][2][NE]
  auto bound_words = [&](int q, int to, int from) { return mw + (((size_t)q * G + to) * G + from) * NM; };
  auto edge_words = [&](int q, int i, int side) { return ew + (((size_t)q * G + i) * 2 + side) * NE; };
  if (G > 1) {
    for (int i = threadIdx.x; i < 2 * G; i += blockDim.x)
#pragma unroll
      for (int n = 0; n < NM; n += 2) put_words2(bound_words(i / G, i % G, b) + n, 0, 0, 0);
    for (int i = threadIdx.x; i < 4 * NE; i += blockDim.x)
      put_word(edge_words(i / (2 * NE), b, (i / NE) & 1) + i % NE, 0, 0);
    __threadfence();
  }
  const StepCtl sc = block_step_ctl(ctl);       // ends with a block barrier
  if (!(sc.dt > 0.0) || S.stall) return;
  R* const U = sc.cur ? bufB : bufA;
  const P<R> k(kp);
  Clock<R> ck;
  ck.start(sc.t, vload(&ctl->t_end), StepDt<R>(sc).dt, vload(&ctl->last) != 0);
  ck.dt_last = sc.dt;
  const long long nsteps0 = vload(&ctl->nsteps);
  int done = 0;

  // the warp's window: cells c0 - 2 .. c0 + cnt + 1 at positions 0 .. cnt + 3
  const int c0 = live ? (int)((int64_t)gw * N / wtot) : 0;
  const int cnt = live ? (int)((int64_t)(gw + 1) * N / wtot) - c0 : 0;
  const bool first = gw == 0, final_w = gw == wtot - 1;
  R X[CPL][4];
  bool own[CPL];
  int rh[CPL];                                  // right halo cell (0 or 1) of the position
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    const int pos = CPL * lane + c;
    own[c] = live && pos >= 2 && pos < 2 + cnt;
    rh[c] = live ? pos - (2 + cnt) : 2;
    const int j = c0 - 2 + (pos < cnt + 3 ? pos : cnt + 3);
    if (j < 0 && k.bc_lo == BC_DRIVEN) {
      double u[4];
      drive_state(kp, ((double)j + 0.5) * kp.h, ck.t, u);
#pragma unroll
      for (int f = 0; f < 4; ++f) X[c][f] = (R)(PP == 3 ? u[f] - kp.ref[f] : u[f]);
    } else {
      bool flip;
      const int i = bc_index(j, N, k.bc_lo, k.bc_hi, flip);
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const R v = U[f * N + i];
        X[c][f] = (f == 1 && flip) ? -v : v;
      }
    }
  }
  // where the halo cells come from after a step: 0 shared memory, 1 another
  // block's words, 2 the boundary
  const int lsrc = first ? (kp.bc_lo == BC_PERIODIC ? (G > 1 ? 1 : 0) : 2) : (w == 0 ? 1 : 0);
  const int rsrc = final_w ? (kp.bc_hi == BC_PERIODIC ? (G > 1 ? 1 : 0) : 2) : (w == lw ? 1 : 0);
  const int lwarp = w == 0 ? lw : w - 1, rwarp = w == lw ? 0 : w + 1;
  const int lblk = b == 0 ? G - 1 : b - 1, rblk = b == G - 1 ? 0 : b + 1;
  // warps that fetch the other blocks' cells while warp 0 waits for the bounds
  const bool lfetch = G > 1 && w == (W > 1 ? 1 : 0) && !(b == 0 && kp.bc_lo != BC_PERIODIC);
  const bool rfetch = G > 1 && w == W - 1 && !(b == G - 1 && kp.bc_hi != BC_PERIODIC);

  // A driven boundary's two ghost cells, by lane: cell lane / 4, field lane % 4
  // (one double sincos per step instead of one per cell, and no envelope or
  // field after another: 65536 cells in the perturbation layout 7.3 -> 5.5 us)
  const bool driven = first && kp.bc_lo == BC_DRIVEN;
  const int df = lane & 3;
  const DriveCell dcell(kp, ((double)((lane >> 2 & 1) - 2) + 0.5) * kp.h);
  const double dbase = kp.drv_base[df], dre = kp.drv_are[df], dim = kp.drv_aim[df];

  for (int s = 1;; ++s) {
    const int q = s & 1;
    const uint32_t tag = ((sc.gen << 17) | (uint32_t)s) << 1;
    const StepDt<R> sd(kp, ck.dt);
    // the other parity's word: last used in step s - 1, which is behind a
    // barrier, and next in step s + 1, which is behind this step's
    if (threadIdx.x == 0) S.word[q ^ 1] = 0.0f;
    Acc<R> acc(&S.word[q]);
    if (live) window_step<PP, LIM, SRC>(k, X, own, sd, acc);
    // publish the first and last two cells, then the bounds
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      const int pos = CPL * lane + c;
      if (own[c]) {
        const int pf = pos - 2, pl = pos - cnt;
        if (pf < 2) {
#pragma unroll
          for (int f = 0; f < 4; ++f) {
            S.edge[q][w][0][pf][f] = X[c][f];
            if (G > 1 && w == 0)
#pragma unroll
              for (int i = 0; i < NW; ++i)
                put_word(edge_words(q, b, 0) + (pf * 4 + f) * NW + i, tag, word_of(X[c][f], i));
          }
        }
        if (pl >= 0) {
#pragma unroll
          for (int f = 0; f < 4; ++f) {
            S.edge[q][w][1][pl][f] = X[c][f];
            if (G > 1 && w == lw)
#pragma unroll
              for (int i = 0; i < NW; ++i)
                put_word(edge_words(q, b, 1) + (pl * 4 + f) * NW + i, tag, word_of(X[c][f], i));
          }
        }
      }
    }
    {
      const R m = warp_max(acc.smax), a = SRC != 0 ? warp_max(acc.akey) : (R)-INFINITY;
      const uint32_t f = __reduce_or_sync(0xffffffffu, acc.flags);
      if (lane == 0) {
        S.smax[q][w] = m;
        S.akey[q][w] = a;
        S.fl[q][w] = f;
      }
    }
    __syncthreads();
    // the block's maxima
    const bool in = lane < W;
    R smax = warp_max(in ? S.smax[q][in ? lane : 0] : (R)0);
    R akey = SRC != 0 ? warp_max(in ? S.akey[q][in ? lane : 0] : (R)-INFINITY) : (R)-INFINITY;
    uint32_t flags = __reduce_or_sync(0xffffffffu, in ? S.fl[q][in ? lane : 0] : 0u);
    if (G > 1) {
      bool ok = true;
      // each warp sends them to 32 blocks ...
      for (int g = w; g * 32 < G; g += W) {
        const int i = g * 32 + lane;
        if (i < G) {
          uint64_t* const p = bound_words(q, i, b);
          const uint32_t tg = tag | (flags ? 1u : 0u);
          if constexpr (NW == 1) {
            put_words2(p, tg, word_of(smax, 0), word_of(akey, 0));
          } else {
            put_words2(p, tg, word_of(smax, 0), word_of(smax, 1));
            put_words2(p + 2, tg, word_of(akey, 0), word_of(akey, 1));
          }
        }
      }
      // ... and waits for those of 32
      for (int g = w; g * 32 < G; g += W) {
        const int i = g * 32 + lane;
        uint64_t x[NM] = {};
        const bool got = wait_words(bound_words(q, b, i < G ? i : 0), i < G, tag, x, kp.stall_polls);
        ok = ok && got;
        R m = (R)0, a = (R)-INFINITY;
        uint32_t f = 0;
        if (got && i < G) {
          uint32_t v[NM];
#pragma unroll
          for (int n = 0; n < NM; ++n) v[n] = (uint32_t)x[n];
          from_words(v, m);
          from_words(v + NW, a);
          f = ((uint32_t)(x[0] >> 32) & 1u) ? FLAG_NONPHYS : 0u;
        }
        __syncwarp();
        m = warp_max(m);
        if (SRC != 0) a = warp_max(a);
        f = __reduce_or_sync(0xffffffffu, f);
        if (lane == 0) {
          S.bmax[g] = m;
          S.bkey[g] = a;
          S.bflags[g] = f;
        }
      }
      if (lfetch && lane < NE) {
        uint64_t x[1] = {0};
        ok = wait_words(edge_words(q, lblk, 1) + lane, true, tag, x, kp.stall_polls) && ok;
        (&S.halo[0][0][0][0])[lane] = (uint32_t)x[0];
      }
      if (rfetch && lane < NE) {
        uint64_t x[1] = {0};
        ok = wait_words(edge_words(q, rblk, 0) + lane, true, tag, x, kp.stall_polls) && ok;
        (&S.halo[1][0][0][0])[lane] = (uint32_t)x[0];
      }
      if (!ok) S.stall = 1;
      if (s == 1) __threadfence();              // step 2's words: after the clears
      __syncthreads();
      if (S.stall) {
        if (threadIdx.x == 0) atomicOr(&ctl->flags, FLAG_STALL);
        if (b == 0 && threadIdx.x == 0) ctl->gen = sc.gen + 1u;
        return;
      }
      smax = S.bmax[0];
      akey = S.bkey[0];
      flags = S.bflags[0];
      for (int g = 1; g * 32 < G; ++g) {
        smax = fmax(smax, S.bmax[g]);
        akey = fmax(akey, S.bkey[g]);
        flags |= S.bflags[g];
      }
    }
    // (the clamp to t_end reads and writes S.t between barriers of its own)
    ck.advance(kp, smax, akey, flags, w == 0, &S.t, false, [](double) { return 0u; });
    done = s;
    if (ck.stop || s >= nmax) break;

    // halo cells of the next step
    if (driven) {                                // warp 0, which keeps t
      double sn, cs;
      dcell.phase(kp, ck.t, sn, cs);
      const double v = dcell.field(dbase, dre, dim, sn, cs);
      const R g = (R)(PP == 3 ? v - kp.ref[df] : v);
#pragma unroll
      for (int c = 0; c < CPL; ++c)
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          const R x = __shfl_sync(0xffffffffu, g, 4 * (CPL * lane + c) + f);
          if (CPL * lane + c < 2) X[c][f] = x;
        }
    }
    if (live) {
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        const int pos = CPL * lane + c;
        if (pos < 2) {
#pragma unroll
          for (int f = 0; f < 4; ++f) {
            if (lsrc == 0) X[c][f] = S.edge[q][lwarp][1][pos][f];
            else if (lsrc == 1) from_words(S.halo[0][pos][f], X[c][f]);
          }
          if (lsrc == 2) {
            if (!driven) {
              // wall: cells 1, 0 with the velocity reversed; outflow: cell 0
              const int m = kp.bc_lo == BC_REFLECT ? 1 - pos : 0;
#pragma unroll
              for (int f = 0; f < 4; ++f) {
                const R v = S.edge[q][w][0][m][f];
                X[c][f] = (f == 1 && kp.bc_lo == BC_REFLECT) ? -v : v;
              }
            }
          }
        }
        if (rh[c] >= 0 && rh[c] < 2) {
#pragma unroll
          for (int f = 0; f < 4; ++f) {
            if (rsrc == 0) X[c][f] = S.edge[q][rwarp][0][rh[c]][f];
            else if (rsrc == 1) from_words(S.halo[1][rh[c]][f], X[c][f]);
            else {
              const int m = kp.bc_hi == BC_REFLECT ? 1 - rh[c] : 1;
              const R v = S.edge[q][w][1][m][f];
              X[c][f] = (f == 1 && kp.bc_hi == BC_REFLECT) ? -v : v;
            }
          }
        }
      }
    }
  }
  // the state goes back where it came from: every block had read its cells
  // before it published step 1
#pragma unroll
  for (int c = 0; c < CPL; ++c)
    if (own[c]) {
      const int j = c0 - 2 + CPL * lane + c;
#pragma unroll
      for (int f = 0; f < 4; ++f) U[f * N + j] = X[c][f];
    }
  if (b == 0 && threadIdx.x == 0) {
    ctl->t = ck.t;
    ctl->dt_cfl = (double)ck.dt_cfl;
    ctl->nsteps = nsteps0 + done;
    ctl->last = ck.last ? 1u : 0u;
    // 0 when the launch began; a block that gave up in the last step has left its
    // cells unwritten and may have raised its flag already
    if (ck.flags) atomicOr(&ctl->flags, ck.flags);
    ctl->gen = sc.gen + 1u;         // every block has read it: each published a step
    set_step_dt<R>(ctl, ck.last ? ck.dt_last : (double)ck.dt, kp);
  }
}

template <typename R, int PP, int LIM>
void* res_src(int src) {
  switch (src) {
    case 0: return (void*)res1d_kernel<R, PP, LIM, 0>;
    case 1: return (void*)res1d_kernel<R, PP, LIM, 1>;
    default: return (void*)res1d_kernel<R, PP, LIM, 2>;
  }
}

template <typename R, int PP>
void* res_pick(const KParams& kp) {
  const int src = kp.frozen ? 0 : (kp.qi_zero ? 1 : 2);
  switch (kp.limiter) {
    case 1: return res_src<R, PP, 1>(src);
    case 2: return res_src<R, PP, 2>(src);
    default: return res_src<R, PP, 0>(src);
  }
}

}  // namespace

// The kernels per arithmetic, each in its own translation unit.
void* res1d_pick_f(const KParams& kp);
void* res1d_pick_pc(const KParams& kp);
void* res1d_pick_ps(const KParams& kp);
void* res1d_pick_d(const KParams& kp);

}  // namespace sv
