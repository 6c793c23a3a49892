// sv_internal.h -- declarations shared by the host runtime and the kernel
// translation units of libsv.so (not part of the public C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "sv_march.h"

namespace sv {

struct KParams;
struct Ctl;

enum { PREC_FP32 = 0, PREC_FP64 = 1, PREC_FP32_P64 = 2, PREC_FP32_PC = 3, PREC_FP32_PS = 4 };

// A kernel launch; pdl = with the programmatic stream-serialization
// attribute (for kernels that call pdl_wait before reading what the previous
// kernel wrote: the 1D step kernels), as the solver's step graph records them.
inline cudaError_t launch_kernel(const void* fn, dim3 grid, dim3 block, void** args, size_t smem,
                                 cudaStream_t st, bool pdl) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = pdl ? attr : nullptr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

// 1D fused step (sv_step1d.cu)
int step1d_grid(const KParams& kp, int precision);
cudaError_t step1d_launch(int precision, const KParams& kp, void* a, void* b, Ctl* ctl, int64_t N,
                          int grid, cudaStream_t st, bool pdl = false);

// Float 1D MUSCL-Hancock step on block tiles (sv_tile1d.cu), grids of at
// least kTile1dMinCells cells; precision PREC_FP32, PREC_FP32_PC or PREC_FP32_PS
constexpr int64_t kTile1dMinCells = 4096;
// var = 10 * (cell pairs per thread) + (blocks per SM of the register budget):
// 13, 12 or 22
int tile1d_grid(const KParams& kp, int precision, int var);
cudaError_t tile1d_launch(const KParams& kp, int precision, int var, void* a, void* b, Ctl* ctl,
                          int64_t N, int grid, cudaStream_t st, bool pdl = false);

// 1D persistent loop of up to nmax steps (sv_loop1d.cu); grid 0 = unavailable
int loop1d_grid(const KParams& kp, int precision, int64_t N);
cudaError_t loop1d_launch(int precision, const KParams& kp, void* a, void* b, Ctl* ctl, int64_t N,
                          int grid, int64_t nmax, cudaStream_t st);

// 1D steps with the state resident in registers (sv_res1d.cu).  Blocks of up to
// kResWarps* warps (the register file at 102 / 255 registers a thread; float
// 182400 cells, double 34048 on 152 SMs), at most one per SM and kResBlocks in
// all.  A grid of at most kResLone* warps runs in one block, without the
// exchange through L2 (0.6 us of a step); a larger one in blocks of at least
// kResFew* warps: fewer warps leave schedulers idle, more share them.  Float, us
// per step by warps per block: 1000 cells 2.50 (2) 2.21 (4) 2.35 (8) 2.75 (all
// 17); 20000 cells 3.09 (4) 3.21 (8) 3.51 (16).  Double: 1600 cells 9.49 (2, 3)
// 9.95 (4) 16.1 (8: two warps per FP64 unit).
constexpr int kResBlocks = 160;
constexpr int kResWarpsF = 20, kResWarpsD = 8;
constexpr int kResLoneF = 12, kResLoneD = 4;
constexpr int kResFewF = 4, kResFewD = 3;
struct ResShape {
  int blocks, threads, wtot;    // blocks 0: not available for this grid
};
ResShape res1d_shape(const KParams& kp, int precision, int64_t N);
size_t res1d_word_bytes(int precision, int64_t N);   // exchange words, zeroed once
cudaError_t res1d_launch(int precision, const KParams& kp, void* a, void* b, Ctl* ctl,
                         uint64_t* words, int64_t N, const ResShape& r, int nmax,
                         cudaStream_t st);

// 1D Heun (SSP-RK2) stages (sv_heun1d.cu); stage 1 or 2
int heun1d_grid(const KParams& kp, int precision);
cudaError_t heun1d_launch(int precision, int stage, const KParams& kp, void* a, void* b, Ctl* ctl,
                          int64_t N, int grid, cudaStream_t st);

// 2D / 3D fused steps (sv_stepnd.cu); n[] cells per axis; nseg = segments the
// marching axis is cut into, from march_segments (sv_march.h)
int stepnd_grid(int dim, int precision, const KParams& kp);
MarchShape stepnd_shape(int dim, int precision);
cudaError_t stepnd_launch(int dim, int precision, const KParams& kp, void* a, void* b, Ctl* ctl,
                          const int64_t* n, int nseg, cudaStream_t st);
// The float 2D step marching plane pairs (sv_stepnd_pair.cu), precision
// PREC_FP32 or PREC_FP32_PC; n == nullptr sets the kernels' shared-memory limits
MarchShape stepnd_pair_shape();
cudaError_t stepnd_pair_launch(int dim, int precision, const KParams& kp, void* a, void* b, Ctl* ctl,
                               const int64_t* n, int nseg, cudaStream_t st);

// The float 3D step with the fields in packed pairs (sv_stepnd3f.cu),
// precision PREC_FP32, PREC_FP32_PC or PREC_FP32_PS (the last compiled in
// sv_stepnd3f_ps.cu); n == nullptr sets the kernels' shared-memory limits
MarchShape stepnd3f_shape();
cudaError_t stepnd3f_launch(int precision, const KParams& kp, void* a, void* b, Ctl* ctl,
                            const int64_t* n, int nseg, cudaStream_t st);
cudaError_t stepnd3f_launch_ps(const KParams& kp, void* a, void* b, Ctl* ctl, const int64_t* n,
                               int nseg, cudaStream_t st);

// Batched sweep kernels of 256 (sv_batch.cu) and 128 (sv_batch128.cu) threads
void* batch_pick256(int limiter, int precision);
void* batch_pick128(int limiter, int precision);

// Utility kernels (sv_util.cu)
cudaError_t ctl_reset_launch(Ctl* ctl, double t, cudaStream_t st);
cudaError_t dt_reduce_launch(int precision, int dim, const KParams& kp, const void* a,
                             const void* b, Ctl* ctl, int64_t ncell, cudaStream_t st);
cudaError_t set_target_launch(int precision, Ctl* ctl, double t_end, const KParams& kp,
                              cudaStream_t st);
// Upload of a host-format (double or float) full state: conversion, and the dt of
// the state it leaves in the same pass (kp.ref: the reference state that the
// perturbation layout PREC_FP32_PS subtracts).
cudaError_t upload_launch(int precision, int dim, const KParams& kp, const double* src, void* a,
                          void* b, Ctl* ctl, int64_t ncell, cudaStream_t st);
cudaError_t upload_launch(int precision, int dim, const KParams& kp, const float* src, void* a,
                          void* b, Ctl* ctl, int64_t ncell, cudaStream_t st);
// Device state -> host format; `ref` as kp.ref above.
cudaError_t from_state_launch(int precision, const void* a, const void* b, const Ctl* ctl,
                              double* dst, int64_t count, cudaStream_t st, const double* ref,
                              int nf);
cudaError_t from_state_launch(int precision, const void* a, const void* b, const Ctl* ctl,
                              float* dst, int64_t count, cudaStream_t st, const double* ref,
                              int nf);
// Exact copy of the current state buffer's `bytes` to (save) or from `other`.
cudaError_t raw_state_launch(void* a, void* b, const Ctl* ctl, void* other, int64_t bytes,
                             bool save, cudaStream_t st);
cudaError_t sums_launch(int precision, const void* a, const void* b, const Ctl* ctl, int nf,
                        int64_t ncell, double* partial, int nblocks, double* out,
                        cudaStream_t st);
int sums_blocks();
cudaError_t fill_equilibrium_launch(int precision, void* a, int nf, int64_t ncell, double gamma,
                                    double ev0, cudaStream_t st);

}  // namespace sv
