// sv_cluster.cuh -- exchange between the blocks of a thread-block cluster: the
// barrier, stores to another block's shared memory and the maxima of the dt
// bounds.
#pragma once

#include "sv_window1d.cuh"

namespace sv {

namespace {

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Barrier of the run's blocks: orders their shared and global stores before
// the loads behind it.
__device__ __forceinline__ void cluster_bar(int C) {
  if (C == 1) __syncthreads();
  else
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Store a 4-byte word to the same shared variable of block `rank`.
__device__ __forceinline__ void put_cluster(const void* var, int rank, uint32_t v) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(var);
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(r), "r"(v) : "memory");
}
__device__ __forceinline__ void put_cluster(const float* var, int rank, float v) {
  put_cluster((const void*)var, rank, __float_as_uint(v));
}
__device__ __forceinline__ void put_cluster(const double* var, int rank, double v) {
  put_cluster((const void*)var, rank, (uint32_t)__double2loint(v));
  put_cluster((const char*)var + 4, rank, (uint32_t)__double2hiint(v));
}

// Room for the maxima of every warp of the cluster, by step parity.
template <typename R, int NS>
struct ClusterMax {
  R smax[2][NS], akey[2][NS];
  uint32_t fl[2][NS];
};

// The cluster's maxima of what each thread has folded: every warp tells every
// block, one barrier, every warp reads them all.
template <typename R, int NS>
__device__ __forceinline__ void cluster_max(ClusterMax<R, NS>& S, int q, int rank, int C, int W,
                                            const Acc<R>& acc, R& smax, R& akey, uint32_t& flags) {
  const int lane = threadIdx.x & 31, me = rank * W + (threadIdx.x >> 5);
  const R m = warp_max(acc.smax), a = warp_max(acc.akey);
  const uint32_t f = __reduce_or_sync(0xffffffffu, acc.flags);
  if (lane < C) {
    put_cluster(&S.smax[q][me], lane, m);
    put_cluster(&S.akey[q][me], lane, a);
    put_cluster((const void*)&S.fl[q][me], lane, f);
  }
  cluster_bar(C);
  smax = (R)0;
  akey = (R)-INFINITY;
  flags = 0;
  for (int i = lane; i < C * W; i += 32) {
    smax = fmax(smax, S.smax[q][i]);
    akey = fmax(akey, S.akey[q][i]);
    flags |= S.fl[q][i];
  }
  smax = warp_max(smax);
  akey = warp_max(akey);
  flags = __reduce_or_sync(0xffffffffu, flags);
}

}  // namespace

}  // namespace sv
