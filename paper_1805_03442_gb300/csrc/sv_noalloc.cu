// sv_noalloc.cu -- a 1D step entry point that allocates no memory at all.
//
// The regular solver (sv_init) owns a device block that holds, besides the
// two state buffers, a small control block: time, dt, the eq.-16 reduction
// keys and the completion ticket that the fused step kernel updates.  Some
// callers cannot provide that block through cudaMalloc: processes whose device
// memory is a fixed pool handed out at start-up and that forbid allocation
// afterwards, and hosts that must not allocate on their stepping path (a
// device allocation can synchronise the device and takes unbounded time).
// For them sv_step1d_noalloc takes the state buffers from the caller and
// keeps the control block in the file-scope array below instead.
//
// The array is a static __device__ object: every GPU that loads libsv.so
// holds it (SV_NOALLOC_SCRATCH_BYTES) until the process exits.  Host code
// cannot use its name as a device address; its address is obtained with
// cudaGetSymbolAddress, once per device, the first time the entry point runs
// on that device, together with the launch grid of each step kernel it uses.
#include <mutex>

#include "sv.h"
#include "sv_cluster.cuh"
#include "sv_internal.h"
#include "sv_window1d.cuh"

namespace sv {

namespace {

// The whole call on a grid that one cluster holds: dt of U_in, one step to
// U_out, and what the call returns, in one launch (reset, dt reduction and step
// were three launches, 17 us on 1000 cells).  Each warp keeps its window in
// registers from the first bound to the store.
constexpr int kOnceCluster = 8;      // blocks of a cluster every device supports
template <typename R> struct OnceWarps;
template <> struct OnceWarps<float> { static constexpr int N = 20; };
template <> struct OnceWarps<double> { static constexpr int N = 8; };

struct OnceResult {
  double t;            // the dt taken (0: none)
  uint32_t flags;
};

template <typename R, int PP, int LIM, int SRC>
__global__ void __launch_bounds__(OnceWarps<R>::N * 32, 1)
once1d_kernel(const KParams kp, const R* Uin, R* Uout, OnceResult* out, int n, int wtot, int C) {
  constexpr int CPL = Win<R>::CPL;
  __shared__ ClusterMax<R, OnceWarps<R>::N * kOnceCluster> S;
  __shared__ float s_word[2];
  const int W = blockDim.x >> 5, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int rank = C == 1 ? 0 : (int)cluster_rank(), gw = rank * W + w;
  if (threadIdx.x == 0) s_word[0] = s_word[1] = 0.0f;
  cluster_bar(C);                    // every block of the cluster has started
  const P<R> k(kp);
  const bool live = gw < wtot;
  const int c0 = live ? (int)((int64_t)gw * n / wtot) : 0;
  const int cnt = live ? (int)((int64_t)(gw + 1) * n / wtot) - c0 : 0;
  R X[CPL][4];
  bool own[CPL];
  Acc<R> acc(&s_word[0]);
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    const int pos = CPL * lane + c;
    own[c] = live && pos >= 2 && pos < 2 + cnt;
    const int j = wrap(c0 - 2 + (pos < cnt + 3 ? pos : cnt + 3), n);
#pragma unroll
    for (int f = 0; f < 4; ++f) X[c][f] = Uin[f * n + j];
  }
#pragma unroll
  for (int c = 0; c < CPL; ++c)
    if (own[c]) cell_bound<PP, 1>(k, X[c], acc);
  R smax, akey;
  uint32_t flags;
  cluster_max(S, 0, rank, C, W, acc, smax, akey, flags);
  const R dt = step_rule(kp, smax, akey, flags);
  if (flags == 0) {                  // the same in every thread
    const StepDt<R> sd(kp, dt);
    Acc<R> next(&s_word[1]);
    if (live) window_step<PP, LIM, SRC>(k, X, own, sd, next);
#pragma unroll
    for (int c = 0; c < CPL; ++c)
      if (own[c])
#pragma unroll
        for (int f = 0; f < 4; ++f) Uout[f * n + c0 - 2 + CPL * lane + c] = X[c][f];
    cluster_max(S, 1, rank, C, W, next, smax, akey, flags);
    step_rule(kp, smax, akey, flags);  // flags of the state reached
    if (gw == 0 && lane == 0) *out = {(double)dt, flags};
  } else if (gw == 0 && lane == 0) {
    *out = {0.0, flags};
  }
}

template <typename R, int PP, int LIM>
void* once_src(int src) {
  switch (src) {
    case 0: return (void*)once1d_kernel<R, PP, LIM, 0>;
    case 1: return (void*)once1d_kernel<R, PP, LIM, 1>;
    default: return (void*)once1d_kernel<R, PP, LIM, 2>;
  }
}
template <typename R, int PP>
void* once_pick(const KParams& k) {
  const int src = k.frozen ? 0 : (k.qi_zero ? 1 : 2);
  switch (k.limiter) {
    case 1: return once_src<R, PP, 1>(src);
    case 2: return once_src<R, PP, 2>(src);
    default: return once_src<R, PP, 0>(src);
  }
}

// Most cells one cluster holds.
int64_t once_cells(int precision) {
  return precision == PREC_FP64 ? (int64_t)kOnceCluster * OnceWarps<double>::N * Win<double>::OWN
                                : (int64_t)kOnceCluster * OnceWarps<float>::N * Win<float>::OWN;
}

// One block up to 12 (double: 4) warps, where the cluster's barrier costs more
// than a block's warps crowding its schedulers; then the fewest blocks of about
// 4 warps, in powers of two.
cudaError_t once_launch(int precision, const KParams& kp, const void* in, void* outU,
                        OnceResult* out, int64_t n64, cudaStream_t st) {
  const bool dbl = precision == PREC_FP64;
  const int n = (int)n64, own = dbl ? Win<double>::OWN : Win<float>::OWN;
  int wtot = (n + own - 1) / own, C = 1;
  if (wtot > (dbl ? 4 : 12))
    while (C < kOnceCluster && 4 * C < wtot) C *= 2;
  const int W = (wtot + C - 1) / C;
  const void* fn = dbl ? once_pick<double, 0>(kp)
                       : (precision == PREC_FP32 ? once_pick<float, 0>(kp) : once_pick<float, 2>(kp));
  void* args[] = {(void*)&kp, &in, &outU, &out, (void*)&n, &wtot, &C};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)C);
  cfg.blockDim = dim3((unsigned)W * 32);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = C > 1 ? 1 : 0;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

}  // namespace

}  // namespace sv

namespace {

static __device__ __align__(256) unsigned char g_noalloc_scratch[SV_NOALLOC_SCRATCH_BYTES];

static_assert(sizeof(sv::Ctl) <= SV_NOALLOC_SCRATCH_BYTES, "control block must fit the scratch");

constexpr int kMaxDevices = 64;
constexpr int kKernels = 4 * 3 * 3;   // precision (SV_FP32 .. SV_FP32_PC) x limiter x source
std::mutex g_mutex;
void* g_addr[kMaxDevices] = {};
// The results of a call that waits for them.  Where the GPU shares the host's
// page tables (a coherent link, as on Grace), the kernel stores them here itself
// and the call only waits for the stream: 31 us instead of 37 on 1000 cells with
// a copy of 16 bytes into pageable memory.
alignas(64) sv::OnceResult g_result[kMaxDevices];
int g_direct[kMaxDevices] = {};   // 0: not asked, 1: the GPU can store there, 2: it cannot
int g_grid[kMaxDevices][kKernels] = {};

// Device address of the scratch array and the persistent grid of the step
// kernel of k on the current device (set-up on the first call per device and
// kernel, with that device current; the kernel's shared-memory attribute is
// set then and stays set).
int setup(const sv::KParams& k, int precision, bool once, void** addr, int* grid,
          sv::OnceResult** direct) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return SV_ECUDA;
  if (dev < 0 || dev >= kMaxDevices) return SV_EINVAL;
  const int src = k.frozen ? 0 : (k.qi_zero ? 1 : 2);
  const int kid = (precision * 3 + k.limiter) * 3 + src;
  std::lock_guard<std::mutex> lock(g_mutex);
  if (!g_addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return SV_ECUDA;
    g_addr[dev] = p;
  }
  if (!g_direct[dev]) {
    int pageable = 0, tables = 0;
    cudaDeviceGetAttribute(&pageable, cudaDevAttrPageableMemoryAccess, dev);
    cudaDeviceGetAttribute(&tables, cudaDevAttrPageableMemoryAccessUsesHostPageTables, dev);
    g_direct[dev] = pageable && tables ? 1 : 2;
  }
  *direct = g_direct[dev] == 1 ? &g_result[dev] : nullptr;
  if (!once && g_grid[dev][kid] < 1) {
    const int g = sv::step1d_grid(k, precision);
    if (g < 1) return SV_ECUDA;
    g_grid[dev][kid] = g;
  }
  *addr = g_addr[dev];
  *grid = g_grid[dev][kid];
  return SV_OK;
}

// Whether the byte ranges [a, a + n) and [b, b + n) share a byte.
bool overlap(const void* a, const void* b, uint64_t n) {
  const uint64_t x = (uint64_t)(uintptr_t)a, y = (uint64_t)(uintptr_t)b;
  return x < y ? y - x < n : x - y < n;
}

}  // namespace

extern "C" int sv_step1d_noalloc(const sv_params* p, int64_t n, double L, const void* U_in,
                                 void* U_out, double* dt_used, uint32_t* flags,
                                 void* cuda_stream) {
  using namespace sv;
  if (!p || !U_in || !U_out) return SV_EINVAL;
  if (n > SV_NOALLOC_MAX_CELLS) return SV_ESIZE;
  if (n < 1 || !(L > 0.0)) return SV_EINVAL;
  if (!(p->gamma > 1.0) || !(p->cfl > 0.0) || !(p->c_tau > 0.0) || !(p->tau0 > 0.0) ||
      p->limiter < SV_MINMOD || p->limiter > SV_MC || p->precision < SV_FP32 ||
      p->precision > SV_FP32_PC || p->method != SV_HANCOCK)   // not the perturbation layout
    return SV_EINVAL;
  // the fused step reads U_in's neighbours after other blocks wrote U_out:
  // the two 4 n-element buffers must not share a byte
  const uint64_t span = 4ull * (uint64_t)n * (p->precision == SV_FP64 ? 8u : 4u);
  if (overlap(U_in, U_out, span)) return SV_EINVAL;
  cudaStream_t st = (cudaStream_t)cuda_stream;

  KParams k;
  memset(&k, 0, sizeof k);
  k.gamma = p->gamma;
  k.g1 = p->gamma - 1.0;
  k.Ck = p->Ck;
  k.S = p->S;
  k.frozen = isinf(p->tau0) ? 1 : 0;
  k.tau0 = p->tau0;
  k.inv_tau0 = k.frozen ? 0.0 : 1.0 / p->tau0;
  k.Q0 = k.frozen ? 0.0 : p->S / p->tau0;
  k.tau_rho = p->tau_rho;
  k.tau_T = p->tau_T;
  k.Q_rho = p->Q_rho;
  k.Q_T = p->Q_T;
  k.I_rho = p->I_rho;
  k.I_T = p->I_T;
  k.qi_zero = (p->Q_rho == 0.0 && p->Q_T == 0.0 && p->I_rho == 0.0 && p->I_T == 0.0) ? 1 : 0;
  k.h = L / (double)n;
  k.cfl = p->cfl;
  k.c_tau = p->c_tau;
  k.limiter = p->limiter;
  kparams_finish(k);

  void* scratch = nullptr;
  int grid = 0;
  const bool once = n <= once_cells(p->precision);
  OnceResult* direct = nullptr;
  const int rc = setup(k, p->precision, once, &scratch, &grid, &direct);
  if (rc != SV_OK) return rc;
  Ctl* ctl = (Ctl*)scratch;
  if (once) {
    if (!dt_used && !flags) direct = nullptr;
    OnceResult* out = direct ? direct : (OnceResult*)scratch;
    if (once_launch(p->precision, k, U_in, U_out, out, n, st) != cudaSuccess) return SV_ECUDA;
    if (dt_used || flags) {
      OnceResult r;
      if (!direct &&
          cudaMemcpyAsync(&r, out, sizeof r, cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return SV_ECUDA;
      if (cudaStreamSynchronize(st) != cudaSuccess) return SV_ECUDA;
      if (direct) {
        const volatile OnceResult* v = direct;
        r.t = v->t;
        r.flags = v->flags;
      }
      if (dt_used) *dt_used = r.t;
      if (flags) *flags = r.flags;
    }
    return SV_OK;
  }
  // The scratch keeps whatever the previous call left: reset the control block
  // (time 0, ticket 0, reduction keys, flags, current buffer = U_in) first.
  if (ctl_reset_launch(ctl, 0.0, st) != cudaSuccess) return SV_ECUDA;
  // dt of U_in (eq. 16 with the tau cap), then one fused step U_in -> U_out
  if (dt_reduce_launch(p->precision, 1, k, U_in, U_out, ctl, n, st) != cudaSuccess)
    return SV_ECUDA;
  if (step1d_launch(p->precision, k, (void*)U_in, U_out, ctl, n, grid, st) != cudaSuccess)
    return SV_ECUDA;
  if (dt_used || flags) {
    // the step advanced the control block's time from 0 by the dt it took
    Ctl c;
    if (cudaMemcpyAsync(&c, ctl, sizeof c, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return SV_ECUDA;
    if (dt_used) *dt_used = c.t;
    if (flags) *flags = c.flags;
  }
  return SV_OK;
}
