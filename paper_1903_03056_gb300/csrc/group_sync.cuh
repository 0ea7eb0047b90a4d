// Cluster and plane-group synchronisation, and the L2-only workspace accesses of the collision
// kernels.
#pragma once

#include <cuda_runtime.h>

#include "fft_line.cuh"

namespace dgfs {

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// the two halves of the cluster barrier (CL > 1)
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int CL>
__device__ __forceinline__ void cluster_sync() {
  if constexpr (CL == 1) {
    __syncthreads();
  } else {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
                 "barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

// read an int in the shared memory of the cluster's rank-0 CTA (distributed shared memory)
__device__ __forceinline__ int ld_rank0(const int* local) {
  const unsigned addr = static_cast<unsigned>(__cvta_generic_to_shared(local));
  unsigned remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(remote) : "r"(addr));
  int v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(remote) : "memory");
  return v;
}

// workspace loads/stores go to L2 only: the data is written by other SMs of the cluster
template <typename T> __device__ __forceinline__ C<T> ld2(const C<T>* p) { return __ldcg(p); }
template <typename T> __device__ __forceinline__ void st2(C<T>* p, C<T> v) { __stcg(p, v); }

// Hint that [p, p + bytes) (16-byte aligned, a multiple of 16 bytes) is read soon: one bulk
// prefetch into L2, so the loads that follow meet L2 rather than DRAM latency.  The workspace
// of all clusters exceeds L2, so a volume written in one phase is partly evicted before it is
// read in the next.
__device__ __forceinline__ void prefetch_l2(const void* p, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Barrier of one plane group.  A group of N threads that divides a warp lives inside one warp
// and synchronises only that warp.  Otherwise SG = lcm(N, 32) / N consecutive groups form a
// warp-aligned super-group that synchronises on its own named barrier (ids 1, 2, ...), so
// super-groups run independently; when the groups of a CTA do not split into super-groups
// the CTA barrier is used (every group then runs the same control flow).
constexpr int gcd_int(int a, int b) { return b == 0 ? a : gcd_int(b, a % b); }

template <int N, int GP>
struct GroupSync {
  static constexpr int LCM = N / gcd_int(N, 32) * 32;
  static constexpr int SG = LCM / N;  // plane groups per super-group
  static constexpr bool WARP = N <= 32 && 32 % N == 0;
  static constexpr bool NAMED = !WARP && GP % SG == 0 && GP / SG <= 15;
};

template <int N, int GP>
__device__ __forceinline__ void group_sync() {
  using S = GroupSync<N, GP>;
  if constexpr (S::WARP) {
    __syncwarp();
  } else if constexpr (S::NAMED) {
    const int sg = int(threadIdx.x) / S::LCM;
    asm volatile("bar.sync %0, %1;" ::"r"(1 + sg), "n"(S::LCM) : "memory");
  } else {
    __syncthreads();
  }
}

}  // namespace dgfs
