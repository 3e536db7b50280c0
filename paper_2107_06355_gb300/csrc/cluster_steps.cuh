// Small lattices: all steps of a call in one launch, one thread-block cluster per lattice.
//
// A lattice of a few thousand nodes leaves most of the chip idle however its two passes
// are launched, and a step's time is that of two launches and two dependent passes: 10.7 us
// for 256 x 4 nodes with plain launches, 7.9 with dependent ones (dependent_launch.cuh), of
// which the arithmetic's latency is about 4.5. Here the cluster's blocks share the nodes, and
// the hardware cluster barrier (release / acquire, no spinning in software) separates the
// passes: 6.7 us (an interface at T_r = 0.6, some of whose nodes take the double-precision
// collision; 5.6 at T_r = 0.8, where few do). The per-node arithmetic is the step kernels', so
// the results are bitwise theirs.
#pragma once

#include <cuda_runtime.h>

#include "step_device.cuh"

namespace pplbm {
namespace {

constexpr int kClusterThreads = 256;

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ unsigned cluster_blocks() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}

// nsteps steps of one lattice; sa[p] reads buffer p. Every thread of the cluster calls it.
template <int KIND, bool ST>
__device__ __forceinline__ void cluster_steps(const StepArgs* sa, int parity0, int nsteps) {
  const int n = (int)sa->n, nx = sa->nx;
  const int stride = cluster_blocks() * blockDim.x, first = cluster_rank() * blockDim.x + threadIdx.x;
  const float inv = 1.0f / (float)nx;  // row of node i: exact for n < 2^22
  for (int s = 0; s < nsteps; ++s) {
    const StepArgs& a = sa[(parity0 + s) & 1];
    for (int i = first; i < n; i += stride) rho_psi_node<KIND>(a, a.f_in, i);
    cluster_barrier();
    for (int i = first; i < n; i += stride) {
      const int y = (int)(((float)i + 0.5f) * inv);
      collide_node<KIND, false, ST>(a, i - y * nx, y, nullptr, nullptr, nullptr, nullptr);
    }
    cluster_barrier();
  }
}

inline cudaLaunchConfig_t cluster_config(int lattices, ClusterShape shape, cudaLaunchAttribute* at, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(lattices * shape.blocks));
  cfg.blockDim = dim3((unsigned)shape.threads);
  cfg.stream = s;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = (unsigned)shape.blocks;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

// One thread per node: 128 threads per block up to 2,048 nodes and 256 above, in a power of
// two of blocks; {0, 0} (the step kernels) for lattices of more than `limit` nodes, for more
// than 65,536 in all, where the device cannot hold such a cluster, or too few of them at a time
// (clusters_pay).
// The lines, us per step, clusters / two launches: one lattice of 256 to 2,048 nodes 6.7 / 7.9
// (two-phase 7.7 / 9.0, with the source 8.5 / 9.5, six rates 9.4 / 10.5), of 3,072 or 4,096
// 8.5 / 7.9 (10.1 / 9.0, 11.6 / 9.5, 14.8 / 10.5), so 2,048 (kClusterNodes). The batched
// kernels look their lattice up: 24 lattices of 400 nodes 6.5 / 10.3, 100 of them 7.8 / 14.4,
// 48 of 1,024 7.6 / 11.8, 32 of 2,048 8.5 / 14.0, 6 of 4,096 7.5 / 11.3 and 16 of them 10.3 /
// 14.0, so 4,096 there (kClusterBatchNodes), and 2,048 with six rates.
constexpr int kClusterNodes = 2048, kClusterBatchNodes = 4096;

inline ClusterShape cluster_shape(const void* kernel, int limit, int64_t max_nodes, int64_t all_nodes, int lattices) {
  ClusterShape shape{1, max_nodes <= 2048 ? 128 : 256};
  if (max_nodes > limit || all_nodes > 65536) return ClusterShape{0, 0};
  while ((int64_t)shape.blocks * shape.threads < max_nodes) shape.blocks *= 2;
  if (shape.blocks > 8 && cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    return ClusterShape{0, 0};
  }
  cudaLaunchAttribute at[1];
  const cudaLaunchConfig_t cfg = cluster_config(lattices, shape, at, nullptr);
  int fit = 0;
  if (cudaOccupancyMaxActiveClusters(&fit, kernel, &cfg) != cudaSuccess) cudaGetLastError();
  return clusters_pay(shape.blocks, lattices, fit) ? shape : ClusterShape{0, 0};
}

// launches `lattices` clusters of the given shape
inline cudaError_t launch_clusters(const void* kernel, int lattices, ClusterShape shape, void** args, cudaStream_t s) {
  cudaLaunchAttribute at[1];
  const cudaLaunchConfig_t cfg = cluster_config(lattices, shape, at, s);
  return cudaLaunchKernelExC(&cfg, kernel, args);
}

}  // namespace
}  // namespace pplbm
