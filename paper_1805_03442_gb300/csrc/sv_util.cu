// sv_util.cu -- small kernels of the runtime: control-block reset, the
// eq.-16 dt reduction of an uploaded state, the t_end clamp, host I/O
// conversion and the compensated conservation sums.
#include "sv_internal.h"
#include "sv_reduce.cuh"
#include "sv_pertnd.cuh"

namespace sv {

constexpr int NTU = 256;

__global__ void ctl_reset_kernel(Ctl* ctl, double t) {
  ctl->t = t;
  clear_step_dt(ctl);
  ctl->dt_cfl = 0.0;
  ctl->t_end = INFINITY;
  ctl->nsteps = 0;
  ctl->cur = 0;
  ctl->last = 0;
  ctl->flags = 0;
  ctl->ticket = 0;
  ctl->gen += 1u;      // words of a resident launch that stalled are not the next one's
  ctl->smax_key = key_of(0.0);
  ctl->tau_key = key_of(-INFINITY);
}

cudaError_t ctl_reset_launch(Ctl* ctl, double t, cudaStream_t st) {
  ctl_reset_kernel<<<1, 1, 0, st>>>(ctl, t);
  return cudaGetLastError();
}

// Sets the target time and re-clamps the pending dt (same rule as the
// step finalize: the step that would reach or pass t_end lands on it).
template <typename R>
__global__ void set_target_kernel(Ctl* ctl, double t_end, const KParams kp) {
  const double t = ctl->t, dt = ctl->dt_cfl;
  ctl->t_end = t_end;
  uint32_t last = 0;
  double dtn = dt;
  if (ctl->flags || !(t < t_end)) {
    dtn = 0.0;
  } else if (dt >= t_end - t) {
    dtn = t_end - t;
    last = 1;
  }
  set_step_dt<R>(ctl, dtn, kp);
  ctl->last = last;
}

cudaError_t set_target_launch(int precision, Ctl* ctl, double t_end, const KParams& kp,
                              cudaStream_t st) {
  if (precision == PREC_FP64)
    set_target_kernel<double><<<1, 1, 0, st>>>(ctl, t_end, kp);
  else
    set_target_kernel<float><<<1, 1, 0, st>>>(ctl, t_end, kp);
  return cudaGetLastError();
}

// Eq. 16 bound of one state, folded into acc.
template <typename R, int PP, int DIM>
__device__ __forceinline__ void fold_bound(const P<R>& k, const R (&u)[DIM + 3], Acc<R>& acc) {
  if constexpr (PP == 3 || std::is_same<R, double>::value) {
    // the perturbation layout, and double
    if constexpr (DIM == 1) cell_bound<PP, 1>(k, u, acc);
    else if constexpr (PP == 3) psn::bound<DIM, 1>(k, u, acc.smax, acc.akey, acc.flags);
    else d64::bound<DIM, 1>(k, u, acc);
  } else {
    const R ir = Ar<R>::rcp(u[0]);
    R kin2 = 0, v2 = 0;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      const R v = u[1 + d] * ir;
      kin2 = fmaf(u[1 + d], v, kin2);
      v2 = fmaf(v, v, v2);
    }
    const R vmag = DIM == 1 ? fabsf(u[1] * ir) : speed_of(v2);
    cfl_cell<PP, 1>(k, u[0], kin2, vmag, u[1 + DIM], u[2 + DIM], acc.smax, acc.akey, acc.flags);
  }
}

// dt of the current state (no step): same per-cell bound and finalize as the
// step kernels.
template <typename R, int PP, int DIM>
__global__ void __launch_bounds__(NTU) dt_reduce_kernel(const KParams kp, const R* a, const R* b,
                                                        Ctl* ctl, int64_t ncell) {
  __shared__ float s_word;
  if (threadIdx.x == 0) s_word = 0.0f;
  __syncthreads();
  const R* U = vload(&ctl->cur) ? b : a;
  const P<R> k(kp);
  Acc<R> acc(&s_word);
  for (int64_t i = (int64_t)blockIdx.x * NTU + threadIdx.x; i < ncell;
       i += (int64_t)gridDim.x * NTU) {
    R u[DIM + 3];
#pragma unroll
    for (int f = 0; f < DIM + 3; ++f) u[f] = U[f * ncell + i];
    fold_bound<R, PP, DIM>(k, u, acc);
  }
  reduce_and_finalize<R, NTU>(ctl, kp, acc.smax, acc.akey, acc.flags, false);
}

static int grid_small(int64_t count) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int64_t g = (count + NTU - 1) / NTU;
  if (g > 4LL * sms) g = 4LL * sms;
  return g < 1 ? 1 : (int)g;
}

template <typename R, int PP>
void dt_reduce_dim(int dim, const KParams& kp, const void* a, const void* b, Ctl* ctl,
                   int64_t ncell, cudaStream_t st) {
  const int g = grid_small(ncell);
  const R *x = (const R*)a, *y = (const R*)b;
  if (dim == 1) dt_reduce_kernel<R, PP, 1><<<g, NTU, 0, st>>>(kp, x, y, ctl, ncell);
  else if (dim == 2) dt_reduce_kernel<R, PP, 2><<<g, NTU, 0, st>>>(kp, x, y, ctl, ncell);
  else dt_reduce_kernel<R, PP, 3><<<g, NTU, 0, st>>>(kp, x, y, ctl, ncell);
}

cudaError_t dt_reduce_launch(int precision, int dim, const KParams& kp, const void* a,
                             const void* b, Ctl* ctl, int64_t ncell, cudaStream_t st) {
  switch (precision) {
    case PREC_FP64: dt_reduce_dim<double, 0>(dim, kp, a, b, ctl, ncell, st); break;
    case PREC_FP32_P64:
    case PREC_FP32_PC: dt_reduce_dim<float, 2>(dim, kp, a, b, ctl, ncell, st); break;
    case PREC_FP32_PS: dt_reduce_dim<float, 3>(dim, kp, a, b, ctl, ncell, st); break;
    default: dt_reduce_dim<float, 0>(dim, kp, a, b, ctl, ncell, st);
  }
  return cudaGetLastError();
}

// The perturbation layout (SV_FP32_PS) holds (float)(U - ref[f]) of field f, the
// difference taken in double; nf = 4, 5 or 6 fields.
struct RefN {
  double v[6];
};

RefN ref_of(const double* ref, int nf) {
  RefN r{};
  const double four[4] = {ref[0], ref[1], ref[2], ref[3]};
  for (int f = 0; f < nf; ++f) r.v[f] = ref_field(four, f, nf);
  return r;
}

// V consecutive elements in accesses of at most 16 bytes.
template <int V, typename T>
__device__ __forceinline__ void load_v(const T* p, T (&v)[V]) {
  if constexpr (std::is_same<T, float>::value && V == 4) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else if constexpr (std::is_same<T, float>::value) {
    const float2 q = *reinterpret_cast<const float2*>(p);
    v[0] = q.x; v[1] = q.y;
  } else {
#pragma unroll
    for (int i = 0; i < V; i += 2) {
      const double2 q = *reinterpret_cast<const double2*>(p + i);
      v[i] = q.x; v[i + 1] = q.y;
    }
  }
}
template <int V, typename T>
__device__ __forceinline__ void store_v(T* p, const T (&v)[V]) {
  if constexpr (std::is_same<T, float>::value && V == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else if constexpr (std::is_same<T, float>::value) {
    *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
  } else {
#pragma unroll
    for (int i = 0; i < V; i += 2)
      *reinterpret_cast<double2*>(p + i) = make_double2(v[i], v[i + 1]);
  }
}
// Host-format (double or float) -> state conversion of an upload, with the dt of
// the state it leaves.  `src` is a device staging buffer or the device view of
// mapped pinned host memory (then the kernel itself moves the bytes over the
// host link, which bounds it).  A thread takes as many consecutive cells as 16
// bytes of the host format hold, all fields, and bounds them from registers.
// A second pass over the state for the bound and 8-byte accesses took, ms,
// against now and a plain copy: 512^3 float 16.7 / 15.3 / 15.2, 8192^2 7.08 / 6.37 / 6.35.
// Fields that are not all aligned for that (odd cell counts) keep the two
// passes (to_state_kernel, dt_reduce_kernel): a cell at a time here, 4-byte
// accesses over the link, took 376 us at 4194301 cells, the two passes 350.
template <bool PS, typename R, typename H>
__device__ __forceinline__ R to_state(H v, double ref) {
  return PS ? (R)((double)v - ref) : (R)v;
}

template <typename H, typename R, int PP, int DIM>
__global__ void __launch_bounds__(NTU)
upload_kernel(const KParams kp, const H* __restrict__ src, R* __restrict__ a, R* __restrict__ b,
              Ctl* ctl, int64_t ncell, RefN ref) {
  constexpr int NF = DIM + 3;
  __shared__ float s_word;
  if (threadIdx.x == 0) s_word = 0.0f;
  __syncthreads();
  R* __restrict__ U = vload(&ctl->cur) ? b : a;
  const P<R> k(kp);
  Acc<R> acc(&s_word);
  const int64_t i0 = (int64_t)blockIdx.x * NTU + threadIdx.x, di = (int64_t)gridDim.x * NTU;
  constexpr int V = 16 / sizeof(H);
  for (int64_t i = V * i0; i < ncell; i += V * di) {
    H h[NF][V];
    R u[NF][V];
#pragma unroll
    for (int f = 0; f < NF; ++f) load_v<V>(src + f * ncell + i, h[f]);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
#pragma unroll
      for (int c = 0; c < V; ++c) u[f][c] = to_state<PP == 3, R>(h[f][c], ref.v[f]);
      store_v<V>(U + f * ncell + i, u[f]);
    }
#pragma unroll
    for (int c = 0; c < V; ++c) {
      R v[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f) v[f] = u[f][c];
      fold_bound<R, PP, DIM>(k, v, acc);
    }
  }
  reduce_and_finalize<R, NTU>(ctl, kp, acc.smax, acc.akey, acc.flags, false);
}

// Elements before the first 128-byte boundary of p (at most n).
template <typename T>
__device__ __forceinline__ int64_t head_of(const T* p, int64_t n) {
  const int64_t h = (int64_t)((128 - ((uintptr_t)p & 127)) & 127) / (int64_t)sizeof(T);
  return h < n ? h : n;
}

// Host format -> state without the dt, and state -> host format of a download.  A
// lane's accesses on the host's side are single ones of 16 bytes from the first
// line boundary on (two of them 32 bytes apart per lane halved the rate of
// a double download, 199 -> 410 us for 32 MB; rows begun at a 16-byte boundary
// inside a line took 306 us instead of 282 at 3000001 cells); those of the state, whose rows
// need not be aligned to the host's, are elements.  Fields are alike but for the
// reference state of the perturbation layout (PS), which takes one row of
// blocks per field; otherwise n counts the elements of all.
template <typename H, typename R, bool PS>
__global__ void __launch_bounds__(NTU)
to_state_kernel(const H* src, R* a, R* b, const Ctl* ctl, int64_t n, RefN ref) {
  const int f = PS ? blockIdx.y : 0;
  R* const U = (vload(&ctl->cur) ? b : a) + f * n;
  const double r = ref.v[f];
  const H* const in = src + f * n;
  constexpr int V = 16 / sizeof(H);
  const int64_t i0 = (int64_t)blockIdx.x * NTU + threadIdx.x, di = (int64_t)gridDim.x * NTU;
  const int64_t head = head_of(in, n), nv = head + (n - head) / V * V;
  if (i0 < head) U[i0] = to_state<PS, R>(in[i0], r);
  for (int64_t i = head + V * i0; i < nv; i += V * di) {
    H h[V];
    load_v<V>(in + i, h);
#pragma unroll
    for (int c = 0; c < V; ++c) U[i + c] = to_state<PS, R>(h[c], r);
  }
  if (nv + i0 < n) U[nv + i0] = to_state<PS, R>(in[nv + i0], r);
}

template <typename H, typename R, bool PS>
__global__ void __launch_bounds__(NTU)
from_state_kernel(const R* a, const R* b, const Ctl* ctl, H* dst, int64_t n, RefN ref) {
  const int f = PS ? blockIdx.y : 0;
  const R* const U = (vload(&ctl->cur) ? b : a) + f * n;
  const double r = ref.v[f];
  H* const out = dst + f * n;
  auto host = [&](R v) { return PS ? (H)(r + (double)v) : (H)v; };
  constexpr int V = 16 / sizeof(H);
  const int64_t i0 = (int64_t)blockIdx.x * NTU + threadIdx.x, di = (int64_t)gridDim.x * NTU;
  const int64_t head = head_of(out, n), nv = head + (n - head) / V * V;
  if (i0 < head) out[i0] = host(U[i0]);
  for (int64_t i = head + V * i0; i < nv; i += V * di) {
    H h[V];
#pragma unroll
    for (int c = 0; c < V; ++c) h[c] = host(U[i + c]);
    store_v<V>(out + i, h);
  }
  if (nv + i0 < n) out[nv + i0] = host(U[nv + i0]);
}

// Raw copies of the current state buffer (`words` 4-byte words) to / from
// `other` (the autotuner's exact save and restore).
__global__ void raw_state_kernel(uint32_t* a, uint32_t* b, const Ctl* ctl, uint32_t* other,
                                 int64_t words, bool save) {
  uint32_t* U = vload(&ctl->cur) ? b : a;
  for (int64_t i = (int64_t)blockIdx.x * NTU + threadIdx.x; i < words;
       i += (int64_t)gridDim.x * NTU) {
    if (save) other[i] = U[i];
    else U[i] = other[i];
  }
}

cudaError_t raw_state_launch(void* a, void* b, const Ctl* ctl, void* other, int64_t bytes,
                             bool save, cudaStream_t st) {
  const int64_t words = bytes / 4;
  raw_state_kernel<<<grid_small(words), NTU, 0, st>>>((uint32_t*)a, (uint32_t*)b, ctl,
                                                      (uint32_t*)other, words, save);
  return cudaGetLastError();
}

template <typename H, typename R, int PP>
void upload_dim(int dim, const KParams& kp, const H* src, void* a, void* b, Ctl* ctl, int64_t ncell,
                cudaStream_t st) {
  const int nf = dim + 3;
  const RefN ref = ref_of(kp.ref, nf);
  R *x = (R*)a, *y = (R*)b;
  if (((uintptr_t)src | (uintptr_t)a | (uintptr_t)b) % 16 != 0 || ncell % (16 / sizeof(H)) != 0) {
    const int64_t n = PP == 3 ? ncell : nf * ncell;
    const dim3 g(grid_small((n + 3) / 4), PP == 3 ? nf : 1);
    to_state_kernel<H, R, PP == 3><<<g, NTU, 0, st>>>(src, x, y, ctl, n, ref);
    dt_reduce_dim<R, PP>(dim, kp, a, b, ctl, ncell, st);
    return;
  }
  const int g = grid_small((ncell + 3) / 4);
  if (dim == 1) upload_kernel<H, R, PP, 1><<<g, NTU, 0, st>>>(kp, src, x, y, ctl, ncell, ref);
  else if (dim == 2) upload_kernel<H, R, PP, 2><<<g, NTU, 0, st>>>(kp, src, x, y, ctl, ncell, ref);
  else upload_kernel<H, R, PP, 3><<<g, NTU, 0, st>>>(kp, src, x, y, ctl, ncell, ref);
}

template <typename H>
cudaError_t upload_impl(int precision, int dim, const KParams& kp, const H* src, void* a, void* b,
                        Ctl* ctl, int64_t ncell, cudaStream_t st) {
  switch (precision) {
    case PREC_FP64: upload_dim<H, double, 0>(dim, kp, src, a, b, ctl, ncell, st); break;
    case PREC_FP32_P64:
    case PREC_FP32_PC: upload_dim<H, float, 2>(dim, kp, src, a, b, ctl, ncell, st); break;
    case PREC_FP32_PS: upload_dim<H, float, 3>(dim, kp, src, a, b, ctl, ncell, st); break;
    default: upload_dim<H, float, 0>(dim, kp, src, a, b, ctl, ncell, st);
  }
  return cudaGetLastError();
}

template <typename H>
cudaError_t from_state_impl(int precision, const void* a, const void* b, const Ctl* ctl, H* dst,
                            int64_t count, cudaStream_t st, const double* ref, int nf) {
  const RefN r = ref_of(ref, nf);
  const int64_t ncell = count / nf;
  if (precision == PREC_FP32_PS)
    from_state_kernel<H, float, true><<<dim3(grid_small((ncell + 3) / 4), nf), NTU, 0, st>>>(
        (const float*)a, (const float*)b, ctl, dst, ncell, r);
  else if (precision == PREC_FP64)
    from_state_kernel<H, double, false><<<grid_small((count + 3) / 4), NTU, 0, st>>>(
        (const double*)a, (const double*)b, ctl, dst, count, r);
  else
    from_state_kernel<H, float, false><<<grid_small((count + 3) / 4), NTU, 0, st>>>(
        (const float*)a, (const float*)b, ctl, dst, count, r);
  return cudaGetLastError();
}

cudaError_t upload_launch(int precision, int dim, const KParams& kp, const double* src, void* a,
                          void* b, Ctl* ctl, int64_t ncell, cudaStream_t st) {
  return upload_impl(precision, dim, kp, src, a, b, ctl, ncell, st);
}
cudaError_t upload_launch(int precision, int dim, const KParams& kp, const float* src, void* a,
                          void* b, Ctl* ctl, int64_t ncell, cudaStream_t st) {
  return upload_impl(precision, dim, kp, src, a, b, ctl, ncell, st);
}
cudaError_t from_state_launch(int precision, const void* a, const void* b, const Ctl* ctl,
                              double* dst, int64_t count, cudaStream_t st, const double* ref,
                              int nf) {
  return from_state_impl<double>(precision, a, b, ctl, dst, count, st, ref, nf);
}
cudaError_t from_state_launch(int precision, const void* a, const void* b, const Ctl* ctl,
                              float* dst, int64_t count, cudaStream_t st, const double* ref,
                              int nf) {
  return from_state_impl<float>(precision, a, b, ctl, dst, count, st, ref, nf);
}

// Uniform equilibrium rho = p = 1, v = 0, E_nu = ev0 into buffer a.
template <typename R>
__global__ void fill_equilibrium_kernel(R* a, int nf, int64_t ncell, double gamma, double ev0) {
  for (int64_t i = (int64_t)blockIdx.x * NTU + threadIdx.x; i < (int64_t)nf * ncell;
       i += (int64_t)gridDim.x * NTU) {
    const int f = (int)(i / ncell);
    double v = 0.0;
    if (f == 0) v = 1.0;
    else if (f == nf - 2) v = 1.0 / (gamma - 1.0) + ev0;
    else if (f == nf - 1) v = ev0;
    a[i] = (R)v;
  }
}

cudaError_t fill_equilibrium_launch(int precision, void* a, int nf, int64_t ncell, double gamma,
                                    double ev0, cudaStream_t st) {
  const int g = grid_small((int64_t)nf * ncell);
  if (precision == PREC_FP32_PS)      // the equilibrium is the layout's reference: all zero
    return cudaMemsetAsync(a, 0, sizeof(float) * (size_t)nf * (size_t)ncell, st);
  if (precision == PREC_FP64)
    fill_equilibrium_kernel<double><<<g, NTU, 0, st>>>((double*)a, nf, ncell, gamma, ev0);
  else
    fill_equilibrium_kernel<float><<<g, NTU, 0, st>>>((float*)a, nf, ncell, gamma, ev0);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- sums

// Neumaier compensated addition of x into (s, c).
__device__ __forceinline__ void neumaier(double& s, double& c, double x) {
  const double t = s + x;
  if (fabs(s) >= fabs(x)) c += (s - t) + x;
  else c += (x - t) + s;
  s = t;
}

constexpr int SUM_BLOCKS = 512;
int sums_blocks() { return SUM_BLOCKS; }

// Pass 1: per block and field, a compensated partial (sum, compensation).
template <typename R>
__global__ void __launch_bounds__(NTU) sums_kernel(const R* a, const R* b, const Ctl* ctl, int nf,
                                                   int64_t ncell, double* partial) {
  const R* U = vload(&ctl->cur) ? b : a;
  __shared__ double sh_s[NTU], sh_c[NTU];
  for (int f = 0; f < nf; ++f) {
    double s = 0.0, c = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * NTU + threadIdx.x; i < ncell;
         i += (int64_t)gridDim.x * NTU)
      neumaier(s, c, (double)U[f * ncell + i]);
    sh_s[threadIdx.x] = s;
    sh_c[threadIdx.x] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
      double S = 0.0, C = 0.0;
      for (int i = 0; i < NTU; ++i) {
        neumaier(S, C, sh_s[i]);
        C += sh_c[i];
      }
      partial[(blockIdx.x * nf + f) * 2 + 0] = S;
      partial[(blockIdx.x * nf + f) * 2 + 1] = C;
    }
    __syncthreads();
  }
}

// Pass 2: fold the block partials (one thread per field).
__global__ void sums_fold_kernel(const double* partial, int nblocks, int nf, double* out) {
  const int f = threadIdx.x;
  if (f >= nf) return;
  double S = 0.0, C = 0.0;
  for (int bk = 0; bk < nblocks; ++bk) {
    neumaier(S, C, partial[(bk * nf + f) * 2 + 0]);
    C += partial[(bk * nf + f) * 2 + 1];
  }
  out[f] = S + C;
}

cudaError_t sums_launch(int precision, const void* a, const void* b, const Ctl* ctl, int nf,
                        int64_t ncell, double* partial, int nblocks, double* out,
                        cudaStream_t st) {
  if (precision == PREC_FP64)
    sums_kernel<double><<<nblocks, NTU, 0, st>>>((const double*)a, (const double*)b, ctl, nf,
                                                 ncell, partial);
  else
    sums_kernel<float><<<nblocks, NTU, 0, st>>>((const float*)a, (const float*)b, ctl, nf, ncell,
                                                partial);
  sums_fold_kernel<<<1, 32, 0, st>>>(partial, nblocks, nf, out);
  return cudaGetLastError();
}

}  // namespace sv
