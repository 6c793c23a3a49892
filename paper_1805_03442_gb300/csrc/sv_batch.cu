// sv_batch.cu -- batched stability sweep: thousands of independent 1D
// periodic runs of uneven sizes and parameters advanced to their own t_end by
// ONE persistent launch.
//
// A cluster of blocks (one block when there are runs enough to fill the device)
// takes a run from a device work queue (the runs of >= 8192 cells first, largest
// first, then the others by decreasing estimated cost, n^2 t_end / L, so that the
// longest runs start first), steps it to completion with the window arithmetic
// of the resident loop (sv_window1d.cuh), and only then takes the next run.  A
// run whose windows fit one per warp keeps its state in registers; a longer one
// streams its windows through L2.  The dt reduction goes through the cluster's
// shared memory with one barrier per step: no grid barrier, no host round trip.
// At sampled times the cluster projects the velocity on the logged Fourier mode
// m,
//   a_m(t) = (1/n) sum_j v_j exp(-i 2 pi m (j + 1/2) / n),
// which is what a growth-rate fit of the linear stage needs.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <numeric>
#include <queue>
#include <vector>

#include "sv_batch_kernel.cuh"

namespace sv {

// Kernels of the two block sizes: 256 threads here, 128 in sv_batch128.cu.
void* batch_pick256(int limiter, int precision) { return bpick<256>(limiter, precision); }

// The states that the runs are at, to page-locked host memory: blockIdx.x over
// the runs, blockIdx.y over parts of one.  A run's block of 4 stride elements is
// a multiple of 128 elements and starts at one.
static __global__ void __launch_bounds__(256) gather_states_kernel(const RunDev* runs, int nruns,
                                                            const unsigned char* a,
                                                            const unsigned char* b,
                                                            unsigned char* host, int esize) {
  for (int i = blockIdx.x; i < nruns; i += gridDim.x) {
    const size_t off = (size_t)runs[i].off * esize;
    const uint4* const src = (const uint4*)((runs[i].cur ? b : a) + off);
    uint4* const dst = (uint4*)(host + off);
    const int n16 = runs[i].stride * 4 * esize / 16;
    for (int j = blockIdx.y * 256 + threadIdx.x; j < n16; j += gridDim.y * 256) dst[j] = src[j];
  }
}

}  // namespace sv

using namespace sv;

struct sv_batch {
  sv_params p;
  int64_t nruns = 0;
  int log_cap = 0;
  int esize = 4;
  bool ps = false;                    // perturbation layout (SV_FP32_PS)
  cudaStream_t stream = nullptr, cap_stream = nullptr;
  void* mem = nullptr;
  bool owns_mem = false;
  void* buf[2] = {nullptr, nullptr};
  RunDev* runs = nullptr;
  int* order = nullptr;
  int* queue = nullptr;
  double* logs = nullptr;
  std::vector<RunDev> host_runs;      // the records as last uploaded
  // Page-locked copies of what a run leaves: its records, logs and states,
  // copied behind the kernel as part of the run (an upload packs its states there
  // too).  Null (the reads then copy from the device each time) beyond
  // kMirrorBytes; `staging` then holds one run's state.  With 256 runs a
  // copy and a wait per read and a pageable upload took 14 of a sweep's 32 ms
  // on the host, now 11 of 28.9.
  RunDev* mirror = nullptr;
  double* mirror_logs = nullptr;
  unsigned char* staging = nullptr;
  void* staging_dev = nullptr;        // its device address
  bool whole = false;                 // staging holds every run's state
  std::vector<int64_t> n;
  int64_t n_max = 0;
  std::vector<int> host_order;        // queue order
  int64_t total_elems = 0;
  int grid = 0;                       // blocks: a multiple of `cluster`
  int cluster = 1;                    // blocks per run
  int nt = 256;                       // threads per run (block size)
  int config = 0;                     // index into kBatchConfigs
  void* fn = nullptr;
  cudaGraphExec_t graph = nullptr;
  int64_t max_steps = 0;
};

namespace {

constexpr size_t kAlignB = 256;
size_t alb(size_t x) { return (x + kAlignB - 1) / kAlignB * kAlignB; }

constexpr size_t kMirrorBytes = (size_t)64 << 20;

struct BLayout {
  size_t state, runs, order, queue, logs, total;
};

// What a step costs besides its rounds of windows, in rounds (1.4 us with the
// device full), for clusters of 1, 2, 4, 8 and 16 blocks: a run that streams its
// windows, and one that keeps its single round in registers.  Measured, us per
// step with every SM full, streaming 2 rounds / resident: 3.86 / 2.16 (1 block),
// 4.29 / 2.40 (2), 4.34 / 2.42 (4), 4.36 / 2.77 (8), 4.59 / 3.08 (16).
constexpr double kBatchLat[5][2] = {{0.8, 0.55}, {1.0, 0.7}, {1.05, 0.73}, {1.1, 0.95}, {1.2, 1.2}};

// Runs of at least this many cells lead the queue (sv_batch_init).
constexpr int64_t kBigRun = 8192;

// With such runs, of the cluster sizes that end the sweep within this factor of
// the best by the estimate, the one that bounds a run at the step cap best: which
// runs get there no estimate foresees, and one of them can outlast the rest.
// 4096 runs of 256-16384 cells, 33 of them capped: 23.5 s with one block per run,
// 19.4 s by this rule (a factor of 1.2 costs at most that where none is).
constexpr double kTailRoom = 1.2;

int64_t stride_of(int64_t n) { return (n + 31) / 32 * 32; }

int check_batch(const sv_params* p, const sv_run* r, int64_t nruns, int log_cap) {
  if (!p || !r || nruns < 1 || nruns > (1 << 30) || log_cap < 0) return SV_EINVAL;
  if (!(p->gamma > 1.0) || !(p->cfl > 0.0) || !(p->c_tau > 0.0)) return SV_EINVAL;
  if (p->limiter < SV_MINMOD || p->limiter > SV_MC) return SV_EINVAL;
  if (p->precision < SV_FP32 || p->precision > SV_FP32_PS) return SV_EINVAL;
  if (p->method != SV_HANCOCK) return SV_EINVAL;
  for (int64_t i = 0; i < nruns; ++i) {
    if (r[i].n < 1 || r[i].n > (1 << 24) || !(r[i].L > 0.0) || !(r[i].tau0 > 0.0) ||
        !(r[i].t_end >= 0.0) || r[i].mode < 0)
      return SV_EINVAL;
  }
  return SV_OK;
}

BLayout blayout(const sv_params* p, const sv_run* r, int64_t nruns, int log_cap) {
  int64_t elems = 0;
  for (int64_t i = 0; i < nruns; ++i) elems += 4 * stride_of(r[i].n);
  const size_t es = p->precision == SV_FP64 ? 8 : 4;
  BLayout L;
  L.state = alb((size_t)elems * es);
  L.runs = alb(sizeof(RunDev) * (size_t)nruns);
  L.order = alb(sizeof(int) * (size_t)nruns);
  L.queue = alb(sizeof(int));
  L.logs = alb(sizeof(double) * 3 * (size_t)log_cap * (size_t)nruns);
  L.total = 2 * L.state + L.runs + L.order + L.queue + L.logs;
  return L;
}

#define SVB_TRY(expr)                        \
  do {                                       \
    cudaError_t e_ = (expr);                 \
    if (e_ != cudaSuccess) return SV_ECUDA;  \
  } while (0)

// The runs' states in the device's format and layout (host: concatenation over
// runs of (4, n_r) field-major blocks; the perturbation layout holds U - ref,
// the difference taken in double).
template <typename R>
void pack_states(const sv_batch* b, const double* host, R* out) {
  for (int64_t i = 0; i < b->nruns; ++i) {
    const int64_t n = b->n[(size_t)i], st = stride_of(n);
    const RunDev& r = b->host_runs[(size_t)i];
    for (int f = 0; f < 4; ++f) {
      const double ref = b->ps ? r.kp.ref[f] : 0.0;
      R* o = out + r.off + f * st;
      for (int64_t j = 0; j < n; ++j) o[j] = (R)(host[j] - ref);
      host += n;
    }
  }
}

int upload(sv_batch* b, const double* host) {
  const size_t bytes = (size_t)b->total_elems * (size_t)b->esize;
  std::vector<unsigned char> tmp;
  if (b->whole) SVB_TRY(cudaStreamSynchronize(b->stream));   // a run may be copying its states there
  else tmp.resize(bytes, 0);
  unsigned char* const packed = b->whole ? b->staging : tmp.data();
  if (b->esize == 8) pack_states(b, host, (double*)packed);
  else pack_states(b, host, (float*)packed);
  SVB_TRY(cudaMemcpyAsync(b->buf[0], packed, bytes, cudaMemcpyHostToDevice, b->stream));
  for (auto& r : b->host_runs) {
    r.t = 0.0;
    r.steps = 0;
    r.flags = 0;
    r.cur = 0;
    r.log_count = 0;
  }
  SVB_TRY(cudaMemcpyAsync(b->runs, b->host_runs.data(), sizeof(RunDev) * b->host_runs.size(),
                          cudaMemcpyHostToDevice, b->stream));
  if (cudaStreamSynchronize(b->stream) != cudaSuccess) return SV_ECUDA;
  if (b->mirror) memcpy(b->mirror, b->host_runs.data(), sizeof(RunDev) * b->host_runs.size());
  return SV_OK;
}

// Launch configurations of the batch kernel (sv_batch_set_config): block size
// per run.  Smaller blocks keep more runs in flight and idle fewer warps on
// small runs; larger ones finish each run sooner.
struct BatchConfig {
  int nt;
  const char* desc;
};
constexpr BatchConfig kBatchConfigs[] = {
    {256, "batch: 256 threads (8 warps) per run, 64-cell chunks, 2 cells per thread"},
    {128, "batch: 128 threads (4 warps) per run, 64-cell chunks, 2 cells per thread"},
};
constexpr int kNumBatchConfigs = (int)(sizeof(kBatchConfigs) / sizeof(kBatchConfigs[0]));

// The launch of `clusters` clusters of C blocks.
struct BatchLaunch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  BatchLaunch(int clusters, int C, int nt, cudaStream_t st) {
    cfg.gridDim = dim3((unsigned)(clusters * C));
    cfg.blockDim = dim3((unsigned)nt);
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = C > 1 ? 1 : 0;
  }
};

// Time of the whole sweep, in rounds, when runs are taken in queue order by
// `groups` groups of `warps` warps each: a step is the rounds of windows its
// busiest warp does and `lat`, the number of steps is estimated by the frozen
// sound speed at rest.
double sweep_time(const sv_batch* b, const std::vector<int>& order, int groups, int warps,
                  const double (&lat)[2]) {
  const int own = b->esize == 8 ? 28 : 60;
  std::priority_queue<double, std::vector<double>, std::greater<double>> free_at;
  for (int i = 0; i < groups && i < (int)order.size(); ++i) free_at.push(0.0);
  double end = 0.0;
  for (int id : order) {
    const RunDev& r = b->host_runs[(size_t)id];
    const int64_t windows = (r.n + own - 1) / own;
    const double rounds = (double)((windows + warps - 1) / warps);
    const double steps = std::max(1.0, std::min((double)b->max_steps,
                                                r.t_end * sqrt(r.kp.gamma) / r.kp.cfl_h));
    const double t = free_at.top() + steps * (rounds + lat[rounds == 1.0 ? 1 : 0]);
    free_at.pop();
    free_at.push(t);
    if (t > end) end = t;
  }
  return end;
}

// Time of the largest run of at least kBigRun cells if its step size collapses and
// it runs to the step cap, in rounds (0: no such run).
double capped_time(const sv_batch* b, int warps, const double (&lat)[2]) {
  if (b->n_max < kBigRun) return 0.0;
  const int own = b->esize == 8 ? 28 : 60;
  const double rounds = (double)(((b->n_max + own - 1) / own + warps - 1) / warps);
  return (double)b->max_steps * (rounds + lat[rounds == 1.0 ? 1 : 0]);
}

// Pick the kernel of configuration c, the blocks per run and the persistent
// grid (host side, outside any capture).
//
// One block per run keeps the device busiest when there are many more runs than
// blocks fit; with fewer, or when a few long runs are left at the end, SMs
// idle while the others step one run each, so a run is given a cluster of 2 to
// 16 blocks, whichever ends the sweep first by sweep_time.  Sweeps in ms, one
// block of a sliding kernel per run (before) / one block / this choice: 256 runs
// of 256-6000 cells 67 / 63 / 17.9 (8 blocks), 400 of 500-4000 38 / 32 / 12.4 (4),
// 2000 of 256-2000 13.1 / 9.2 / 9.2 (1), 8 of 20000-40000 168 / 178 / 17.1 (16).
int apply_config(sv_batch* b, int c) {
  const int nt = kBatchConfigs[c].nt;
  void* fn = nt == 128 ? batch_pick128(b->p.limiter, b->p.precision)
                       : batch_pick256(b->p.limiter, b->p.precision);
  int dev = 0, sms = 0, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, nt, 0) != cudaSuccess)
    return SV_ECUDA;
  struct Choice {
    int groups, cluster;
    double time, tail;
  };
  std::vector<Choice> choices;
  auto weigh = [&](int groups, int C, const double (&lat)[2]) {
    choices.push_back({groups, C, sweep_time(b, b->host_order, groups, C * nt / 32, lat),
                       capped_time(b, C * nt / 32, lat)});
  };
  weigh(sms * (per < 1 ? 1 : per), 1, kBatchLat[0]);
  // 16 blocks are beyond the size every device supports: asked for, and skipped
  // below where it is not available
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    cudaGetLastError();
  for (int C = 2, i = 1; C <= kBatchCluster; C *= 2, ++i) {
    int nc = 0;
    const BatchLaunch l(1, C, nt, nullptr);
    if (cudaOccupancyMaxActiveClusters(&nc, fn, &l.cfg) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    // clusters of 16: half of what the occupancy query says run at once (18
    // asked for: 5.8 us per step, 9: 3.1)
    if (C == 16) nc /= 2;
    if (nc < 1) continue;
    weigh(nc, C, kBatchLat[i]);
  }
  double least = choices[0].time;
  for (const Choice& c : choices) least = std::min(least, c.time);
  Choice pick = {0, 0, 0.0, 0.0};
  for (const Choice& c : choices) {
    if (c.time > least * (b->n_max >= kBigRun ? kTailRoom : 1.0)) continue;
    if (!pick.cluster || c.tail < pick.tail || (c.tail == pick.tail && c.time < pick.time)) pick = c;
  }
  int groups = pick.groups;
  const int cluster = pick.cluster;
  if (b->graph) {
    if (cudaStreamSynchronize(b->stream) != cudaSuccess) return SV_ECUDA;
    cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
  }
  b->fn = fn;
  b->nt = nt;
  b->config = c;
  b->cluster = cluster;
  if ((int64_t)groups > b->nruns) groups = (int)b->nruns;
  b->grid = groups * cluster;
  return SV_OK;
}

size_t log_bytes(const sv_batch* b) {
  return sizeof(double) * 3 * (size_t)b->log_cap * (size_t)b->nruns;
}

cudaError_t launch_batch(sv_batch* b, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(b->queue, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  int nr = (int)b->nruns;
  int lc = b->log_cap;
  int64_t ms = b->max_steps;
  void* args[] = {&b->runs, &b->order, &nr, &b->queue, &b->buf[0], &b->buf[1], &b->logs, &lc, &ms,
                  &b->cluster};
  const BatchLaunch l(b->grid / b->cluster, b->cluster, b->nt, st);
  e = cudaLaunchKernelExC(&l.cfg, b->fn, args);
  if (e == cudaSuccess && b->whole) {
    gather_states_kernel<<<dim3(nr < 1024 ? nr : 1024, 4), 256, 0, st>>>(
        b->runs, nr, (const unsigned char*)b->buf[0], (const unsigned char*)b->buf[1],
        (unsigned char*)b->staging_dev, b->esize);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && b->mirror)
    e = cudaMemcpyAsync(b->mirror, b->runs, sizeof(RunDev) * (size_t)b->nruns,
                        cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess && b->mirror_logs)
    e = cudaMemcpyAsync(b->mirror_logs, b->logs, log_bytes(b), cudaMemcpyDeviceToHost, st);
  return e;
}

// Record of a run, once the stream's work is done.
int read_run(sv_batch* b, int64_t run, RunDev& d) {
  if (!b->mirror)
    SVB_TRY(cudaMemcpyAsync(&d, b->runs + run, sizeof(RunDev), cudaMemcpyDeviceToHost, b->stream));
  SVB_TRY(cudaStreamSynchronize(b->stream));
  if (b->mirror) d = b->mirror[run];
  return SV_OK;
}

template <typename R>
void unpack_state(const R* src, int64_t n, int64_t st, const double* ref, double* out) {
  for (int f = 0; f < 4; ++f)
    for (int64_t j = 0; j < n; ++j) out[f * n + j] = (ref ? ref[f] : 0.0) + (double)src[f * st + j];
}

}  // namespace

extern "C" {

int sv_batch_required_bytes(const sv_params* p, const sv_run* runs, int64_t nruns, int log_cap,
                            size_t* bytes) {
  int rc = check_batch(p, runs, nruns, log_cap);
  if (rc != SV_OK) return rc;
  if (!bytes) return SV_EINVAL;
  *bytes = blayout(p, runs, nruns, log_cap).total;
  return SV_OK;
}

int sv_batch_init(const sv_params* p, const sv_run* runs, int64_t nruns,
                  const double* host_states, int log_cap, int64_t max_steps_per_run,
                  void* cuda_stream, void* device_mem, size_t device_bytes, sv_batch** out) {
  if (!out || !host_states || max_steps_per_run < 1) return SV_EINVAL;
  *out = nullptr;
  int rc = check_batch(p, runs, nruns, log_cap);
  if (rc != SV_OK) return rc;
  const BLayout L = blayout(p, runs, nruns, log_cap);
  if (device_mem && (device_bytes < L.total || ((uintptr_t)device_mem % kAlignB) != 0))
    return SV_ENOMEM;
  sv_batch* b = new (std::nothrow) sv_batch();
  if (!b) return SV_ENOMEM;
  b->p = *p;
  b->nruns = nruns;
  b->log_cap = log_cap;
  b->esize = p->precision == SV_FP64 ? 8 : 4;
  b->ps = p->precision == SV_FP32_PS;
  b->stream = (cudaStream_t)cuda_stream;
  b->max_steps = max_steps_per_run;
  b->host_runs.resize((size_t)nruns);
  b->n.resize((size_t)nruns);
  int64_t off = 0;
  for (int64_t i = 0; i < nruns; ++i) {
    const sv_run& r = runs[i];
    RunDev d;
    memset(&d, 0, sizeof d);
    KParams& k = d.kp;
    k.gamma = p->gamma;
    k.g1 = p->gamma - 1.0;
    k.Ck = p->Ck;
    k.S = r.S;
    k.frozen = isinf(r.tau0) ? 1 : 0;
    k.tau0 = r.tau0;
    k.inv_tau0 = k.frozen ? 0.0 : 1.0 / r.tau0;
    k.Q0 = k.frozen ? 0.0 : r.S / r.tau0;
    k.tau_rho = r.tau_rho;
    k.tau_T = r.tau_T;
    k.Q_rho = r.Q_rho;
    k.Q_T = r.Q_T;
    k.I_rho = r.I_rho;
    k.I_T = r.I_T;
    k.qi_zero = (r.Q_rho == 0.0 && r.Q_T == 0.0 && r.I_rho == 0.0 && r.I_T == 0.0) ? 1 : 0;
    k.h = r.L / (double)r.n;
    k.cfl = p->cfl;
    k.c_tau = p->c_tau;
    k.limiter = p->limiter;
    kparams_finish(k);
    d.src = k.frozen ? 0 : (k.qi_zero ? 1 : 2);
    d.off = off;
    d.n = (int)r.n;
    d.stride = (int)stride_of(r.n);
    d.mode = r.mode;
    d.t_end = r.t_end;
    b->host_runs[(size_t)i] = d;
    b->n[(size_t)i] = r.n;
    b->n_max = std::max<int64_t>(b->n_max, r.n);
    off += 4 * stride_of(r.n);
  }
  b->total_elems = off;

  if (device_mem) b->mem = device_mem;
  else {
    if (cudaMalloc(&b->mem, L.total) != cudaSuccess) {
      delete b;
      return SV_ENOMEM;
    }
    b->owns_mem = true;
  }
  char* m = (char*)b->mem;
  b->buf[0] = m;
  b->buf[1] = m + L.state;
  b->runs = (RunDev*)(m + 2 * L.state);
  b->order = (int*)(m + 2 * L.state + L.runs);
  b->queue = (int*)(m + 2 * L.state + L.runs + L.order);
  b->logs = (double*)(m + 2 * L.state + L.runs + L.order + L.queue);

  // Queue order.  The runs of >= kBigRun cells first, largest first: a run's
  // worst case is the step cap, whose cost grows with n alone, and the few
  // large runs that reach it (their dt collapses long after the start, which
  // no estimate from the initial state foresees) set the sweep's end unless
  // they start early.  Then the others, longest first by the estimated cost
  // n * steps ~ n^2 t_end / L.
  std::vector<int> order((size_t)nruns);
  std::iota(order.begin(), order.end(), 0);
  std::vector<double> cost((size_t)nruns);
  for (int64_t i = 0; i < nruns; ++i)
    cost[(size_t)i] = (double)runs[i].n * (double)runs[i].n * runs[i].t_end / runs[i].L;
  auto big = [&](int i) { return runs[i].n >= kBigRun; };
  std::stable_sort(order.begin(), order.end(), [&](int a, int c) {
    if (big(a) != big(c)) return big(a);
    return big(a) ? runs[a].n > runs[c].n : cost[a] > cost[c];
  });

  b->host_order = order;
  rc = SV_OK;
  if (cudaStreamCreateWithFlags(&b->cap_stream, cudaStreamNonBlocking) != cudaSuccess ||
      cudaMemcpyAsync(b->order, order.data(), sizeof(int) * order.size(), cudaMemcpyHostToDevice,
                      b->stream) != cudaSuccess)
    rc = SV_ECUDA;
  {
    // page-locked copies where they are of a size to keep; without them the
    // reads copy from the device
    int64_t widest = 0;
    for (int64_t n : b->n) widest = std::max(widest, 4 * stride_of(n) * (int64_t)b->esize);
    const size_t rec = sizeof(RunDev) * (size_t)nruns;
    auto lock = [](void** p, size_t bytes) {
      if (bytes == 0 || bytes > kMirrorBytes) return;
      if (cudaMallocHost(p, bytes) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
      }
    };
    lock((void**)&b->mirror, rec);
    if (b->mirror) lock((void**)&b->mirror_logs, log_bytes(b));
    const size_t all = (size_t)b->total_elems * (size_t)b->esize;
    lock((void**)&b->staging, all);
    if (b->staging && cudaHostGetDevicePointer(&b->staging_dev, b->staging, 0) != cudaSuccess) {
      cudaGetLastError();
      cudaFreeHost(b->staging);
      b->staging = nullptr;
    }
    b->whole = b->staging != nullptr;
    if (b->whole) memset(b->staging, 0, all);        // the rows' padding
    else lock((void**)&b->staging, (size_t)widest);
  }
  if (rc == SV_OK) rc = apply_config(b, 0);
  if (rc == SV_OK) rc = upload(b, host_states);
  if (rc != SV_OK) {
    sv_batch_free(b);
    return rc;
  }
  *out = b;
  return SV_OK;
}

int sv_batch_reset(sv_batch* b, const double* host_states) {
  if (!b || !host_states) return SV_EINVAL;
  return upload(b, host_states);
}

int sv_batch_run(sv_batch* b) {
  if (!b) return SV_EINVAL;
  if (!b->graph) {
    cudaGraph_t g = nullptr;
    SVB_TRY(cudaStreamBeginCapture(b->cap_stream, cudaStreamCaptureModeThreadLocal));
    cudaError_t le = launch_batch(b, b->cap_stream);
    cudaError_t ee = cudaStreamEndCapture(b->cap_stream, &g);
    if (le != cudaSuccess || ee != cudaSuccess) {
      if (g) cudaGraphDestroy(g);
      return SV_ECUDA;
    }
    cudaError_t ie = cudaGraphInstantiate(&b->graph, g, 0);
    cudaGraphDestroy(g);
    if (ie != cudaSuccess) {
      b->graph = nullptr;
      return SV_ECUDA;
    }
  }
  SVB_TRY(cudaGraphLaunch(b->graph, b->stream));
  return SV_OK;
}

int sv_batch_sync(sv_batch* b) {
  if (!b) return SV_EINVAL;
  SVB_TRY(cudaStreamSynchronize(b->stream));
  return SV_OK;
}

int sv_batch_read(sv_batch* b, int64_t run, double* host_soa, double* t, int64_t* steps,
                  uint32_t* flags) {
  if (!b || run < 0 || run >= b->nruns) return SV_EINVAL;
  RunDev d;
  int rc = read_run(b, run, d);
  if (rc != SV_OK) return rc;
  if (t) *t = d.t;
  if (steps) *steps = d.steps;
  if (flags) *flags = d.flags;
  if (host_soa) {
    const int64_t n = d.n, st = d.stride;
    const size_t es = (size_t)b->esize;
    const size_t bytes = (size_t)(4 * st) * es;
    std::vector<unsigned char> pageable;
    const unsigned char* tmp = b->staging + (b->whole ? (size_t)d.off * es : 0);
    if (!b->whole) {
      if (!b->staging) pageable.resize(bytes);
      unsigned char* const to = b->staging ? b->staging : pageable.data();
      const char* src = (const char*)b->buf[d.cur ? 1 : 0] + (size_t)d.off * es;
      SVB_TRY(cudaMemcpyAsync(to, src, bytes, cudaMemcpyDeviceToHost, b->stream));
      SVB_TRY(cudaStreamSynchronize(b->stream));
      tmp = to;
    }
    const double* ref = b->ps ? d.kp.ref : nullptr;
    if (es == 8) unpack_state((const double*)tmp, n, st, ref, host_soa);
    else unpack_state((const float*)tmp, n, st, ref, host_soa);
  }
  return SV_OK;
}

int sv_batch_mode_log(sv_batch* b, int64_t run, double* t, double* re, double* im, int64_t cap,
                      int64_t* count) {
  if (!b || run < 0 || run >= b->nruns || cap < 0) return SV_EINVAL;
  RunDev d;
  int rc = read_run(b, run, d);
  if (rc != SV_OK) return rc;
  const int64_t c = std::min<int64_t>(d.log_count, cap);
  if (count) *count = c;
  if (c > 0) {
    const int64_t at = run * (int64_t)b->log_cap * 3;
    std::vector<double> copy;
    const double* tmp = b->mirror_logs + at;
    if (!b->mirror_logs) {
      copy.resize((size_t)c * 3);
      SVB_TRY(cudaMemcpyAsync(copy.data(), b->logs + at, sizeof(double) * copy.size(),
                              cudaMemcpyDeviceToHost, b->stream));
      SVB_TRY(cudaStreamSynchronize(b->stream));
      tmp = copy.data();
    }
    for (int64_t i = 0; i < c; ++i) {
      if (t) t[i] = tmp[(size_t)(3 * i)];
      if (re) re[i] = tmp[(size_t)(3 * i + 1)];
      if (im) im[i] = tmp[(size_t)(3 * i + 2)];
    }
  }
  return SV_OK;
}

int sv_batch_num_configs(sv_batch* b, int* count) {
  if (!b || !count) return SV_EINVAL;
  *count = kNumBatchConfigs;
  return SV_OK;
}

int sv_batch_set_config(sv_batch* b, int index) {
  if (!b || index < 0 || index >= kNumBatchConfigs) return SV_EINVAL;
  return apply_config(b, index);
}

int sv_batch_get_config(sv_batch* b, int* index, char* desc, size_t cap) {
  if (!b) return SV_EINVAL;
  if (index) *index = b->config;
  if (desc && cap > 0) {
    strncpy(desc, kBatchConfigs[b->config].desc, cap - 1);
    desc[cap - 1] = 0;
  }
  return SV_OK;
}

void sv_batch_free(sv_batch* b) {
  if (!b) return;
  if (b->stream || b->mem) cudaStreamSynchronize(b->stream);
  if (b->graph) cudaGraphExecDestroy(b->graph);
  if (b->cap_stream) cudaStreamDestroy(b->cap_stream);
  if (b->mirror) cudaFreeHost(b->mirror);
  if (b->mirror_logs) cudaFreeHost(b->mirror_logs);
  if (b->staging) cudaFreeHost(b->staging);
  if (b->owns_mem && b->mem) cudaFree(b->mem);
  delete b;
}

}  // extern "C"
