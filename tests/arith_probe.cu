// Device arithmetic of the step kernels, function by function, over arrays
// (compiled by test_gpu_arith.py).
#include "sv_pair1d.cuh"
#include "sv_f64.cuh"

using namespace sv;

namespace {

__global__ void f64_kernel(int op, const double* x, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (op == 0) y[i] = d64::rcp(x[i]);
  else if (op == 1) y[i] = d64::sqrt_pos(x[i]);
  else y[i] = op == 2 ? d64::rcp_estimate(x[i]) : d64::rsqrt_estimate(x[i]);
}

// p of (kin2, E, E_nu) by the scalar and by the packed recovery, two states a thread
__global__ void pressure_kernel(const KParams kp, const float* s, float* one, float* two, int n) {
  const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (i + 1 >= n) return;
  const P<float> k(kp);
  for (int c = 0; c < 2; ++c) one[i + c] = pressure<2>(k, s[i + c], s[n + i + c], s[2 * n + i + c]);
  const float* const a[3] = {s + i, s + n + i, s + 2 * n + i};
  const pk::f2 p = pk::pressure<2>(k, pk::pair(a[0][0], a[0][1]), pk::pair(a[1][0], a[1][1]),
                                   pk::pair(a[2][0], a[2][1]));
  two[i] = p.x;
  two[i + 1] = p.y;
}

// Runs `go` between copies of `in` (nin bytes) and `out` (nout bytes).
template <typename F>
int with_buffers(const void* in, size_t nin, void* out, size_t nout, F&& go) {
  void *a = nullptr, *b = nullptr;
  int rc = 1;
  if (cudaMalloc(&a, nin) == cudaSuccess && cudaMalloc(&b, nout) == cudaSuccess &&
      cudaMemcpy(a, in, nin, cudaMemcpyHostToDevice) == cudaSuccess) {
    go(a, b);
    if (cudaGetLastError() == cudaSuccess && cudaMemcpy(out, b, nout, cudaMemcpyDeviceToHost) == cudaSuccess)
      rc = 0;
  }
  cudaFree(a);
  cudaFree(b);
  return rc;
}

}  // namespace

// op 0: d64::rcp, 1: d64::sqrt_pos, 2 and 3: the estimates they begin with, of n doubles.
extern "C" int probe_f64(int op, const double* x, double* y, int n) {
  return with_buffers(x, sizeof(double) * n, y, sizeof(double) * n, [&](void* a, void* b) {
    f64_kernel<<<(n + 255) / 256, 256>>>(op, (const double*)a, (double*)b, n);
  });
}

// Pressures of n (even) states: s holds kin2, E, E_nu of all, p the scalar results
// and then the packed ones.
extern "C" int probe_pressure(double gamma, const float* s, float* p, int n) {
  KParams kp = {};
  kp.gamma = gamma;
  kp.g1 = gamma - 1.0;
  kp.h = kp.cfl = kp.c_tau = kp.tau0 = kp.inv_tau0 = 1.0;
  kparams_finish(kp);
  return with_buffers(s, sizeof(float) * 3 * n, p, sizeof(float) * 2 * n, [&](void* a, void* b) {
    pressure_kernel<<<(n / 2 + 255) / 256, 256>>>(kp, (const float*)a, (float*)b, (float*)b + n, n);
  });
}
