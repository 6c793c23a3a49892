// sv_batch_kernel.cuh -- the persistent kernel of the batched stability sweep
// (see sv_batch.cu), templated on its block size so that each size compiles
// in a translation unit of its own.
#pragma once

#include "sv.h"
#include "sv_internal.h"
#include "sv_cluster.cuh"
#include "sv_window1d.cuh"

namespace sv {

struct RunDev {
  KParams kp;            // per-run parameters (h = L / n)
  int64_t off;           // element offset of the run's block (4 fields x stride)
  int n, stride, mode, log_count;
  int src, pad2;         // source variant of the run (as a single solver would pick it)
  double t, t_end;
  int64_t steps;
  uint32_t flags, cur, pad0, pad1;
};

constexpr uint32_t FLAG_MAXSTEPS = SV_FLAG_MAXSTEPS;

// A run is stepped by a cluster of C blocks (1 <= C <= kBatchCluster).
constexpr int kBatchCluster = 16;

template <typename R, int W>
struct BatchSmem {
  static constexpr int NS = W * kBatchCluster;
  KParams kp;                            // the run's parameters
  ClusterMax<R, NS> mx;
  R sum[2][NS];                          // every warp's part of a logged amplitude
  R halo[2][W][2][2][4];                 // by parity: each warp's halo cells (side, cell, field)
  double t;
  float word[2];                         // speed threshold of the double bound, by parity
  int run;
};

// The window of cells c0 - 2 .. c0 + 62 (float; double: c0 + 29) of a periodic
// run into registers.  Through L2: neighbouring cells are other blocks' work.
__device__ __forceinline__ void load_window(const float* U, int n, int stride, int c0,
                                            float (&X)[2][4]) {
  const int lane = threadIdx.x & 31, j = c0 - 2 + 2 * lane;
  if (c0 >= 2 && c0 + 62 <= n) {               // c0 and stride are even: 8-byte loads
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const float2 v = __ldcg(reinterpret_cast<const float2*>(U + f * stride + j));
      X[0][f] = v.x;
      X[1][f] = v.y;
    }
  } else {
    const int a = wrap(j, n), b = wrap(j + 1, n);
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      X[0][f] = __ldcg(U + f * stride + a);
      X[1][f] = __ldcg(U + f * stride + b);
    }
  }
}
__device__ __forceinline__ void load_window(const double* U, int n, int stride, int c0,
                                            double (&X)[1][4]) {
  const int j = c0 - 2 + (int)(threadIdx.x & 31);
  const int a = j >= 0 && j < n ? j : wrap(j, n);
#pragma unroll
  for (int f = 0; f < 4; ++f) X[0][f] = __ldcg(U + f * stride + a);
}
__device__ __forceinline__ void store_window(float* U, int stride, int c0,
                                             const float (&X)[2][4], const bool (&own)[2]) {
  const int j = c0 - 2 + 2 * (int)(threadIdx.x & 31);
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    if (own[0] && own[1])
      *reinterpret_cast<float2*>(U + f * stride + j) = make_float2(X[0][f], X[1][f]);
    else if (own[0])
      U[f * stride + j] = X[0][f];
  }
}
__device__ __forceinline__ void store_window(double* U, int stride, int c0,
                                             const double (&X)[1][4], const bool (&own)[1]) {
  const int j = c0 - 2 + (int)(threadIdx.x & 31);
#pragma unroll
  for (int f = 0; f < 4; ++f)
    if (own[0]) U[f * stride + j] = X[0][f];
}

// Step run `rd` to its end.  Every thread of the cluster follows the same
// decisions: they all see the same maxima.
template <typename R, int PP, int LIM, int SRC, int W>
__device__ void batch_run(BatchSmem<R, W>& S, RunDev* rd, R* A, R* B, double* lg, int log_cap,
                          int64_t max_steps, int rank, int C) {
  constexpr int CPL = Win<R>::CPL, OWN = Win<R>::OWN;
  const KParams& kp = S.kp;
  const P<R> k(kp);
  const int n = rd->n, stride = rd->stride, mode = rd->mode;
  const double t_end = rd->t_end;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int gw = rank * W + w, nw = C * W;
  const int nwin = (n + OWN - 1) / OWN;
  // contiguous windows [w0, w1) of this warp
  const int w0 = (int)((int64_t)gw * nwin / nw), w1 = (int)((int64_t)(gw + 1) * nwin / nw);
  const double log_dt = log_cap > 1 ? t_end / (double)(log_cap - 1) : INFINITY;
  const bool logs = mode > 0 && log_cap > 0;

  // a_m of the current state (buffer U), a sample of the log
  auto log_mode = [&](const R* U, double t, int slot) {
    R re = 0, im = 0;
    for (int j = gw * 32 + lane; j < n; j += nw * 32) {
      const R r0 = __ldcg(U + j);
      const R v = __ldcg(U + stride + j) / (PP == 3 ? (R)1 + r0 : r0);   // PP 3: perturbations
      R sn, cs;
      const R ph = (R)(2.0 * mode) * ((R)j + (R)0.5) / (R)n;
      if constexpr (sizeof(R) == 4) sincospif(ph, &sn, &cs);
      else sincospi(ph, &sn, &cs);
      re += v * cs;
      im -= v * sn;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      re += __shfl_xor_sync(0xffffffffu, re, o);
      im += __shfl_xor_sync(0xffffffffu, im, o);
    }
    if (lane == 0) {
      put_cluster(&S.sum[0][gw], 0, re);
      put_cluster(&S.sum[1][gw], 0, im);
    }
    cluster_bar(C);
    if (rank == 0 && threadIdx.x == 0) {
      R a = 0, b = 0;
      for (int i = 0; i < nw; ++i) {
        a += S.sum[0][i];
        b += S.sum[1][i];
      }
      lg[3 * slot + 0] = t;
      lg[3 * slot + 1] = (double)a / n;
      lg[3 * slot + 2] = (double)b / n;
    }
    cluster_bar(C);                    // the sums have been read
  };

  // dt of the initial state (same per-cell bound as every step)
  Clock<R> ck;
  int log_count = 0;
  double next_log = INFINITY;
  {
    Acc<R> acc(&S.word[0]);
    for (int j = gw * 32 + lane; j < n; j += nw * 32) {
      const R u[4] = {A[j], A[stride + j], A[2 * stride + j], A[3 * stride + j]};
      cell_bound<PP, 1>(k, u, acc);
    }
    R smax, akey;
    uint32_t flags;
    cluster_max(S.mx, 0, rank, C, W, acc, smax, akey, flags);
    const R d = step_rule(kp, smax, akey, flags);
    const double t = rd->t, r = t_end - t;
    const bool go = flags == 0 && t < t_end;
    const bool last = go && (double)d >= r;
    ck.start(t, t_end, last ? (R)r : d, last);
    ck.flags = flags;
    ck.stop = !go;
    if (logs) {
      log_mode(A, t, 0);
      log_count = 1;
      next_log = t + log_dt;
      if (log_count < log_cap) ck.due(next_log);
    }
  }
  uint32_t cur = 0;
  int64_t steps = 0;
  // the step with these maxima is complete: the clock, and a log sample of
  // the state that `state()` provides in global memory
  auto finish = [&](R smax, R akey, uint32_t flags, auto&& state) {
    ++steps;
    const bool exact =
        ck.advance(kp, smax, akey, flags, w == 0, &S.t, steps >= max_steps, [&](double t) {
          return steps >= max_steps && t < t_end ? FLAG_MAXSTEPS : 0u;
        });
    if (exact && logs && log_count < log_cap && (ck.t >= next_log || ck.stop)) {
      log_mode(state(), ck.t, log_count);
      ++log_count;
      while (next_log <= ck.t) next_log += log_dt;
    }
    if (exact && !ck.stop && logs) ck.due(log_count < log_cap ? next_log : t_end);
  };
  if (nwin <= nw && n >= 2) {
    // one window per warp: the state stays in registers, neighbours' cells come
    // through shared memory with the maxima's barrier, and global memory (A) is
    // written for the log samples and at the end only
    const bool live = gw < nwin;
    const int c0 = live ? (int)((int64_t)gw * n / nwin) : 0;
    const int cnt = live ? (int)((int64_t)(gw + 1) * n / nwin) - c0 : 0;
    const int lg_w = gw == 0 ? nwin - 1 : gw - 1, rg_w = gw == nwin - 1 ? 0 : gw + 1;
    R X[CPL][4];
    bool own[CPL];
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      const int pos = CPL * lane + c;
      own[c] = live && pos >= 2 && pos < 2 + cnt;
      const int j = wrap(c0 - 2 + (pos < cnt + 3 ? pos : cnt + 3), n);
#pragma unroll
      for (int f = 0; f < 4; ++f) X[c][f] = A[f * stride + j];
    }
    auto save = [&]() -> const R* {
#pragma unroll
      for (int c = 0; c < CPL; ++c)
        if (own[c])
#pragma unroll
          for (int f = 0; f < 4; ++f) A[f * stride + c0 - 2 + CPL * lane + c] = X[c][f];
      return A;
    };
    if (!ck.stop) cluster_bar(C);        // every warp has read its cells of A
    while (!ck.stop) {
      const int q = (int)(steps + 1) & 1;
      const StepDt<R> sd(kp, ck.dt);
      if (threadIdx.x == 0) S.word[q ^ 1] = 0.0f;   // as in the resident loop
      Acc<R> acc(&S.word[q]);
      if (live) window_step<PP, LIM, SRC>(k, X, own, sd, acc);
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        const int pos = CPL * lane + c, pf = pos - 2, pl = pos - cnt;
        if (own[c] && pf < 2)            // the left neighbour's right halo
#pragma unroll
          for (int f = 0; f < 4; ++f)
            put_cluster(&S.halo[q][lg_w % W][1][pf][f], lg_w / W, X[c][f]);
        if (own[c] && pl >= 0)           // the right neighbour's left halo
#pragma unroll
          for (int f = 0; f < 4; ++f)
            put_cluster(&S.halo[q][rg_w % W][0][pl][f], rg_w / W, X[c][f]);
      }
      R smax, akey;
      uint32_t flags;
      cluster_max(S.mx, q, rank, C, W, acc, smax, akey, flags);
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        const int pos = CPL * lane + c, rh = pos - (2 + cnt);
        if (live && (pos < 2 || rh == 0 || rh == 1))
#pragma unroll
          for (int f = 0; f < 4; ++f)
            X[c][f] = pos < 2 ? S.halo[q][w][0][pos][f] : S.halo[q][w][1][rh][f];
      }
      finish(smax, akey, flags, [&]() -> const R* {
        const R* a = save();
        cluster_bar(C);
        return a;
      });
    }
    save();
  } else {
    while (!ck.stop) {
      const int q = (int)(steps + 1) & 1;
      const StepDt<R> sd(kp, ck.dt);
      const R* Uin = cur ? B : A;
      R* Uout = cur ? A : B;
      if (threadIdx.x == 0) S.word[q ^ 1] = 0.0f;   // as in the resident loop
      Acc<R> acc(&S.word[q]);
      R X[CPL][4], Y[CPL][4];
      if (w0 < w1) load_window(Uin, n, stride, w0 * OWN, Y);
      for (int i = w0; i < w1; ++i) {
        const int c0 = i * OWN, cnt = min(OWN, n - c0);
        bool own[CPL];
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
          const int pos = CPL * lane + c;
          own[c] = pos >= 2 && pos < 2 + cnt;
#pragma unroll
          for (int f = 0; f < 4; ++f) X[c][f] = Y[c][f];
        }
        if (i + 1 < w1) load_window(Uin, n, stride, c0 + OWN, Y);   // in flight meanwhile
        window_step<PP, LIM, SRC>(k, X, own, sd, acc);
        store_window(Uout, stride, c0, X, own);
      }
      R smax, akey;
      uint32_t flags;
      cluster_max(S.mx, q, rank, C, W, acc, smax, akey, flags);   // orders the stores too
      cur ^= 1u;
      finish(smax, akey, flags, [&]() -> const R* { return cur ? B : A; });
    }
  }
  if (rank == 0 && threadIdx.x == 0) {
    rd->t = ck.t;
    rd->steps = steps;
    rd->flags = ck.flags;
    rd->cur = cur;
    rd->log_count = log_count;
  }
}

// Every run is stepped with the source variant a single 1D solver with the
// same parameters would use (none in the frozen limit, pump = sink for zero
// exponents, general otherwise), chosen per run at run time, so that a batched
// run and a looped solver run execute the same operations.
template <typename R, int PP, int LIM, int NTB, int MINB>
__global__ void __launch_bounds__(NTB, MINB)
batch_kernel(RunDev* __restrict__ runs, const int* __restrict__ order, int nruns,
             int* __restrict__ queue, R* bufA, R* bufB, double* logs, int log_cap,
             int64_t max_steps, int C) {
  constexpr int W = NTB / 32;
  __shared__ BatchSmem<R, W> S;
  const int rank = C == 1 ? 0 : (int)cluster_rank();
  cluster_bar(C);                      // every block of the cluster has started
  for (;;) {
    if (rank == 0 && threadIdx.x < 32) {
      int r = 0;
      if (threadIdx.x == 0) r = atomicAdd(queue, 1);
      r = __shfl_sync(0xffffffffu, r, 0);
      if ((int)threadIdx.x < C) put_cluster((const void*)&S.run, (int)threadIdx.x, (uint32_t)r);
    }
    cluster_bar(C);
    const int qi = S.run;
    if (qi >= nruns) break;
    const int id = order[qi];
    RunDev* rd = runs + id;
    for (int i = threadIdx.x; i < (int)(sizeof(KParams) / 4); i += NTB)
      reinterpret_cast<uint32_t*>(&S.kp)[i] = reinterpret_cast<const uint32_t*>(&rd->kp)[i];
    if (threadIdx.x == 0) S.word[0] = S.word[1] = 0.0f;
    __syncthreads();
    R* const A = bufA + rd->off;
    R* const B = bufB + rd->off;
    double* const lg = logs + (int64_t)id * log_cap * 3;
    if (rd->src == 0) batch_run<R, PP, LIM, 0, W>(S, rd, A, B, lg, log_cap, max_steps, rank, C);
    else if (rd->src == 1) batch_run<R, PP, LIM, 1, W>(S, rd, A, B, lg, log_cap, max_steps, rank, C);
    else batch_run<R, PP, LIM, 2, W>(S, rd, A, B, lg, log_cap, max_steps, rank, C);
    cluster_bar(C);                    // the run's record and this block's memory are free
  }
}

// Kernel of the given block size for (limiter, precision).
template <int NTB, typename R, int PP, int LIM>
struct KB {
  // double and the perturbation layout take the whole register file (one
  // block per SM) rather than spill
  static constexpr int MINB = (sizeof(R) == 8 || PP == 3) ? 1 : 256 / NTB * 2;
  static constexpr auto fn = batch_kernel<R, PP, LIM, NTB, MINB>;
};

template <int NTB, int LIM>
void* bpick_prec(int precision) {
  switch (precision) {
    case PREC_FP64: return (void*)KB<NTB, double, 0, LIM>::fn;
    case PREC_FP32_P64:
    case PREC_FP32_PC: return (void*)KB<NTB, float, 2, LIM>::fn;
    case PREC_FP32_PS: return (void*)KB<NTB, float, 3, LIM>::fn;
    default: return (void*)KB<NTB, float, 0, LIM>::fn;
  }
}
template <int NTB>
void* bpick(int limiter, int precision) {
  switch (limiter) {
    case 1: return bpick_prec<NTB, 1>(precision);
    case 2: return bpick_prec<NTB, 2>(precision);
    default: return bpick_prec<NTB, 0>(precision);
  }
}

}  // namespace sv
