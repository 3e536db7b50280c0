// Device code of the batched engine (batch.cu): the per-instance argument table, the
// work-item kernels of the two passes, the persistent kernel with its bounded grid
// barrier, the per-instance guard, and their launchers. The per-node arithmetic is
// step_device.cuh's, shared with the single-lattice kernels.
#pragma once

#include <cuda_runtime.h>

#include "cluster_steps.cuh"
#include "dependent_launch.cuh"
#include "step_device.cuh"

namespace pplbm {
namespace {

constexpr int kThreads = 256;
constexpr unsigned kSpinLimit = 1u << 24;           // x ~100 ns sleeps: ~1.7 s per barrier wait
constexpr int kErrTimeout = 2;  // batch error word; divergence is flagged per instance

struct BatchInst {
  StepArgs a[2];  // a[p] reads f from buffer p and writes buffer 1 - p
  double* snap;   // density at the previous guard call (one plane)
  int tw, th, log2tw, tiles_x;
  int k1_start, k2_start;
};

struct GridBarrier {
  unsigned int count;
  unsigned int generation;
};

// Bounded grid-wide barrier for a cooperative launch; false if a wait gave up.
__device__ bool grid_barrier(GridBarrier* b, int* err, unsigned spin_limit) {
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned int* gen = &b->generation;
    const unsigned int g = *gen;
    __threadfence();
    const unsigned int arrived = atomicAdd(&b->count, 1u) + 1u;
    if (arrived == gridDim.x) {
      b->count = 0u;
      __threadfence();
      atomicAdd(&b->generation, 1u);
    } else {
      unsigned int it = 0;
      while (*gen == g) {
        if (++it > spin_limit) {
          atomicOr(err, kErrTimeout);
          break;
        }
        __nanosleep(100);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return (*(volatile int*)err & kErrTimeout) == 0;
}

// Copies instance id's StepArgs for `parity` into shared memory (uniform across
// the block, so every later field read is a shared-memory broadcast).
__device__ __forceinline__ void stage_args(const BatchInst* __restrict__ inst, int id, int parity, StepArgs* sa) {
  const unsigned long long* src = reinterpret_cast<const unsigned long long*>(&inst[id].a[parity]);
  unsigned long long* dst = reinterpret_cast<unsigned long long*>(sa);
  for (int k = threadIdx.x; k < (int)(sizeof(StepArgs) / 8); k += blockDim.x) dst[k] = src[k];
  __syncthreads();
}

// A work item is 256 nodes (or a tile of 256), shared by 256 / NT blocks of NT threads; block
// `part` of them. LAUNCHED: one part per block of a dependent launch, which waits for its
// predecessor after its arguments are in (no kernel writes them); otherwise the block takes
// another item afterwards (persistent kernel), so it waits until every thread is done with
// the shared arguments.

// density/psi pass over item w
template <int KIND, int NT, bool LAUNCHED>
__device__ __forceinline__ void batch_rho_psi_item(const BatchInst* __restrict__ inst, const int* __restrict__ owner,
                                                   int w, int part, int parity, StepArgs* sa) {
  const int id = owner[w], local = w - inst[id].k1_start;
  stage_args(inst, id, parity, sa);
  if (LAUNCHED) begin_dependent();
  const int i = local * kThreads + part * NT + threadIdx.x;
  if (i < (int)sa->n) rho_psi_node<KIND>(*sa, sa->f_in, i);
  if (!LAUNCHED) __syncthreads();
}

// collision pass over item w; org: two shared ints for the tile origin, which one thread
// computes per item
template <int KIND, bool ST, int NT, bool LAUNCHED>
__device__ __forceinline__ void batch_collide_item(const BatchInst* __restrict__ inst, const int* __restrict__ owner,
                                                   int w, int part, int parity, StepArgs* sa, int* org) {
  const int id = owner[w];
  const BatchInst& I = inst[id];
  const int tw = I.tw, log2tw = I.log2tw;
  if (threadIdx.x == 0) {
    const int t = w - I.k2_start, tyi = t / I.tiles_x;
    org[0] = (t - tyi * I.tiles_x) * tw;
    org[1] = tyi * I.th;
  }
  stage_args(inst, id, parity, sa);  // ends with a barrier: org is visible
  if (LAUNCHED) begin_dependent();
  const StepArgs& a = *sa;
  const int j = part * NT + (int)threadIdx.x;
  const int x = org[0] + (j & (tw - 1)), y = org[1] + (j >> log2tw);
  if (x < a.nx && y < a.ny) collide_node<KIND, false, ST>(a, x, y, nullptr, nullptr, nullptr, nullptr);
  if (!LAUNCHED) __syncthreads();
}

// Blocks of the two passes' launches. us per step with 256 / 128 / 64 threads: 6 lattices of
// 192^2 22.9 / 20.3 / 20.6 (with the source 26.6 / 22.8 / 22.7), 12 of 256^2 54.2 / 52.4 /
// 53.6, 24 of 400^2 220 / 217 / 221, 35 two-phase 600 x 250 336 / 329 / 337: halves fill a
// small batch's last wave, quarters copy their arguments too often.
constexpr int kBlock = 128, kParts = kThreads / kBlock;

template <int KIND>
__global__ void __launch_bounds__(kBlock) k_batch_rho_psi(const BatchInst* inst, const int* owner, int parity) {
  __shared__ StepArgs sa;
  batch_rho_psi_item<KIND, kBlock, true>(inst, owner, blockIdx.x / kParts, blockIdx.x % kParts, parity, &sa);
}

// ST: some instance has the surface-tension source (kappa != 0); for the others
// kappa_q = 0 makes the source exactly zero, so their results do not change
// Unit relaxation times: 40 resident warps per SM (at most 48 registers); the
// integer-bound collision pass issues faster with the extra warps than it loses to
// the 8-20 bytes of spilled registers. The other kinds keep 32 (they would spill more).
constexpr int collide_min_blocks(int kind) { return kind == kUnitTau ? 5 : 4; }

template <int KIND, bool ST>
__global__ void __launch_bounds__(kBlock, collide_min_blocks(KIND) * kParts)
    k_batch_collide(const BatchInst* inst, const int* owner, int parity) {
  __shared__ StepArgs sa;
  __shared__ int org[2];
  batch_collide_item<KIND, ST, kBlock, true>(inst, owner, blockIdx.x / kParts, blockIdx.x % kParts, parity, &sa, org);
}

// ---- the pipelined plan's mixed kernel ----------------------------------------------

// 8- and 16-byte asynchronous copies global -> shared (cp.async, cached in L1); the
// data is visible to the block after cp_async_wait_all and a barrier. Both addresses
// are aligned to the copy size.
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// A work item of the pipelined plan (int4): x = the instance, with the top bit set for
// a collision tile; for a density item y = its 256-node block within the instance; for
// a collision tile y = log2 of the tile width tw (tile height 256 / tw) and (z, w) the
// tile's origin (x0, y0).
__device__ __forceinline__ bool is_collision_item(const int4& h) { return h.x < 0; }

// Starts the copy of the item's StepArgs (density items: parity p1, collision tiles:
// p2) into dst.
__device__ __forceinline__ void fetch_item_args(const BatchInst* __restrict__ inst, const int4& h, int p1, int p2,
                                                StepArgs* dst) {
  const int id = h.x & 0x7FFFFFFF;
  const unsigned long long* src =
      reinterpret_cast<const unsigned long long*>(&inst[id].a[is_collision_item(h) ? p2 : p1]);
  unsigned long long* d = reinterpret_cast<unsigned long long*>(dst);
  for (int k = threadIdx.x; k < (int)(sizeof(StepArgs) / 8); k += kBlock) cp_async8(d + k, src + k);
}

// The item's pass from its staged arguments
template <int KIND, bool ST>
__device__ __forceinline__ void run_item(const StepArgs& a, const int4& h, int part) {
  const int j = part * kBlock + (int)threadIdx.x;
  if (!is_collision_item(h)) {
    const int i = h.y * kThreads + j;
    if (i < (int)a.n) rho_psi_node<KIND>(a, a.f_in, i);
    return;
  }
  const int log2tw = h.y, tw = 1 << log2tw;
  const int lx = j & (tw - 1), ly = j >> log2tw;
  const int x = h.z + lx, y = h.w + ly;
  if (x < a.nx && y < a.ny) collide_node<KIND, false, ST>(a, x, y, nullptr, nullptr, nullptr, nullptr);
}

// Work items of both passes in one launch (the pipelined plan): density items read
// buffer p1, collision tiles p2. Lattices of one group run their density pass while
// those of the other run their collision pass: both passes are bound by the integer pipe
// (60 % busy run alone), and loads and stores of one overlap the other's arithmetic on
// every SM. The grid is the resident block count G (at most n, the number of parts: kParts
// per item). Block b starts with part b; later parts come in table order from the queue
// counter queue[0] (part G + the counter's old value), taken four ahead: while a block
// computes part k it copies in the arguments and headers of the next ones (rings of 4), so
// that no part waits on its set-up loads. The last block to finish resets queue[0] and the
// finished-block count queue[1] for the next launch. ms per step on 12.9 M nodes with blocks
// of 256 / 128 threads: 0.628 / 0.617; 35 two-phase 600 x 250 0.329 / 0.322.
template <int KIND, bool ST>
__global__ void __launch_bounds__(kBlock, collide_min_blocks(KIND) * kParts)
    k_batch_mixed(const BatchInst* inst, const int4* items, int n, int p1, int p2, unsigned* queue) {
  __shared__ StepArgs sa[4];
  __shared__ int4 hdr[4];
  __shared__ int qi[4];    // the ring slot's part: table index times kParts plus part; -1: none
  __shared__ int part[4];  // of the slot whose header is in hdr
  const int G = gridDim.x;
  if (threadIdx.x == 0) {
    const int t = G + (int)atomicAdd(&queue[0], 3u);
    qi[0] = blockIdx.x;
    qi[1] = t < n ? t : -1;
    qi[2] = t + 1 < n ? t + 1 : -1;
    qi[3] = t + 2 < n ? t + 2 : -1;
  }
  __syncthreads();
  if (threadIdx.x < 3 && qi[threadIdx.x] >= 0) {
    cp_async16(&hdr[threadIdx.x], items + qi[threadIdx.x] / kParts);
    part[threadIdx.x] = qi[threadIdx.x] % kParts;
  }
  cp_async_wait_all();
  __syncthreads();
  fetch_item_args(inst, hdr[0], p1, p2, &sa[0]);
  if (qi[1] >= 0) fetch_item_args(inst, hdr[1], p1, p2, &sa[1]);
  cp_async_wait_all();
  __syncthreads();
  // qi[c] is rewritten during iteration k (thread 0, for item k + 4), so whether item
  // k + 1 exists is read from its slot c1 before the iteration's barrier: slot c1 is
  // not written during iteration k, and every thread reads the same value
  for (int k = 0;; ++k) {
    const int c = k & 3, c1 = (k + 1) & 3, c2 = (k + 2) & 3, c3 = (k + 3) & 3;
    if (qi[c2] >= 0) fetch_item_args(inst, hdr[c2], p1, p2, &sa[c2]);
    int next = -1;
    if (threadIdx.x == 0) {
      if (qi[c3] >= 0) {
        cp_async16(&hdr[c3], items + qi[c3] / kParts);
        part[c3] = qi[c3] % kParts;
      }
      const int t = G + (int)atomicAdd(&queue[0], 1u);
      next = t < n ? t : -1;
    }
    run_item<KIND, ST>(sa[c], hdr[c], part[c]);
    if (threadIdx.x == 0) qi[c] = next;  // slot c now names item k + 4
    const bool more = qi[c1] >= 0;
    cp_async_wait_all();
    __syncthreads();
    if (!more) break;
  }
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&queue[1], 1u) == (unsigned)G - 1u) {
      queue[0] = 0u;
      queue[1] = 0u;
      __threadfence();
    }
  }
}

template <bool ST>
const void* mixed_kernel_t(int kind) {
  switch (kind) {
    case kUnitTau: return (const void*)k_batch_mixed<kUnitTau, ST>;
    case kShearTau: return (const void*)k_batch_mixed<kShearTau, ST>;
    default: return (const void*)k_batch_mixed<kFullMrt, ST>;
  }
}

const void* mixed_kernel(int kind, bool st) { return st ? mixed_kernel_t<true>(kind) : mixed_kernel_t<false>(kind); }

template <int KIND, bool ST>
__global__ void __launch_bounds__(kThreads) k_batch_persistent(const BatchInst* inst, const int* owner1, int n1,
                                                               const int* owner2, int n2, int parity0, long long nsteps,
                                                               GridBarrier* bar, int* err, unsigned spin_limit,
                                                               int absent_block) {
  __shared__ StepArgs sa;
  __shared__ int org[2];
  // barrier self-test only: one block leaves without arriving, so the others' waits run out
  if ((int)blockIdx.x == absent_block) return;
  for (long long s = 0; s < nsteps; ++s) {
    const int parity = (int)((parity0 + s) & 1);
    for (int w = blockIdx.x; w < n1; w += gridDim.x) batch_rho_psi_item<KIND, kThreads, false>(inst, owner1, w, 0, parity, &sa);
    if (!grid_barrier(bar, err, spin_limit)) return;
    for (int w = blockIdx.x; w < n2; w += gridDim.x)
      batch_collide_item<KIND, ST, kThreads, false>(inst, owner2, w, 0, parity, &sa, org);
    if (!grid_barrier(bar, err, spin_limit)) return;
  }
}

// All steps of a call for a batch of small lattices: one cluster per instance.
template <int KIND, bool ST>
__global__ void __launch_bounds__(kClusterThreads) k_batch_cluster(const BatchInst* inst, int parity0, int nsteps) {
  __shared__ StepArgs sa[2];
  const unsigned long long* src =
      reinterpret_cast<const unsigned long long*>(inst[blockIdx.x / cluster_blocks()].a);
  unsigned long long* dst = reinterpret_cast<unsigned long long*>(sa);
  for (int k = threadIdx.x; k < (int)(sizeof(sa) / 8); k += blockDim.x) dst[k] = src[k];
  __syncthreads();
  cluster_steps<KIND, ST>(sa, parity0, nsteps);
}

template <bool ST>
const void* batch_cluster_kernel_t(int kind) {
  switch (kind) {
    case kUnitTau: return (const void*)k_batch_cluster<kUnitTau, ST>;
    case kShearTau: return (const void*)k_batch_cluster<kShearTau, ST>;
    default: return (const void*)k_batch_cluster<kFullMrt, ST>;
  }
}

const void* batch_cluster_kernel(int kind, bool st) {
  return st ? batch_cluster_kernel_t<true>(kind) : batch_cluster_kernel_t<false>(kind);
}

// Guard, pass 1: one block per 256-node work item of the density pass; per block
// (mass, max |u|, bad count, sum |rho - rho'|), reduced in a fixed tree order
// (guard_node, the same terms as the single-lattice guard). Runs after a density
// pass over the current state, so rho, j and psi are those the next step starts
// from. Refreshes the snapshot rho'.
__global__ void __launch_bounds__(kThreads) k_batch_guard_partial(const BatchInst* inst, const int* owner, int parity,
                                                                  const int* snap_valid, double* partials) {
  __shared__ double s[kGuardQ][kThreads];
  const int w = blockIdx.x;
  const int id = owner[w];
  const BatchInst& I = inst[id];
  const StepArgs& a = I.a[parity];
  const int64_t i = (int64_t)(w - I.k1_start) * kThreads + threadIdx.x;
  double v[kGuardQ] = {0.0, 0.0, 0.0, 0.0};
  if (i < a.n) guard_node(a, i, I.snap, snap_valid[id] != 0, v);
  guard_block_reduce<kThreads>(v, s);
  if (threadIdx.x < kGuardQ) partials[kGuardQ * (int64_t)w + threadIdx.x] = s[threadIdx.x][0];
}

// Guard, pass 2: one block per instance over its work items, in a fixed order.
__global__ void __launch_bounds__(kThreads) k_batch_guard_final(const BatchInst* inst, const double* partials,
                                                                int* snap_valid, double* out) {
  __shared__ double s[kGuardQ][kThreads];
  const int id = blockIdx.x;
  const BatchInst& I = inst[id];
  const int nb = (int)((I.a[0].n + kThreads - 1) / kThreads);
  double v[kGuardQ] = {0.0, 0.0, 0.0, 0.0};
  for (int k = threadIdx.x; k < nb; k += kThreads) {
    const double* p = partials + kGuardQ * (int64_t)(I.k1_start + k);
    v[0] += p[0];
    v[1] = fmax(v[1], p[1]);
    v[2] += p[2];
    v[3] += p[3];
  }
  guard_block_reduce<kThreads>(v, s);
  if (threadIdx.x == 0) {
    out[kGuardQ * id + 0] = s[0][0];
    out[kGuardQ * id + 1] = s[1][0];
    out[kGuardQ * id + 2] = s[2][0];
    out[kGuardQ * id + 3] = snap_valid[id] ? s[3][0] / s[0][0] : -1.0;
    snap_valid[id] = 1;
  }
}

template <bool ST>
const void* persistent_kernel_t(int kind) {
  switch (kind) {
    case kUnitTau: return (const void*)k_batch_persistent<kUnitTau, ST>;
    case kShearTau: return (const void*)k_batch_persistent<kShearTau, ST>;
    default: return (const void*)k_batch_persistent<kFullMrt, ST>;
  }
}

const void* persistent_kernel(int kind, bool st) {
  return st ? persistent_kernel_t<true>(kind) : persistent_kernel_t<false>(kind);
}

template <bool ST>
void launch_pair_t(int kind, const BatchInst* inst, const int* o1, int n1, const int* o2, int n2, int parity,
                   cudaStream_t s) {
  switch (kind) {
    case kUnitTau:
      launch_dependent(k_batch_rho_psi<kUnitTau>, n1 * kParts, kBlock, s, inst, o1, parity);
      launch_dependent(k_batch_collide<kUnitTau, ST>, n2 * kParts, kBlock, s, inst, o2, parity);
      break;
    case kShearTau:
      launch_dependent(k_batch_rho_psi<kShearTau>, n1 * kParts, kBlock, s, inst, o1, parity);
      launch_dependent(k_batch_collide<kShearTau, ST>, n2 * kParts, kBlock, s, inst, o2, parity);
      break;
    default:
      launch_dependent(k_batch_rho_psi<kFullMrt>, n1 * kParts, kBlock, s, inst, o1, parity);
      launch_dependent(k_batch_collide<kFullMrt, ST>, n2 * kParts, kBlock, s, inst, o2, parity);
      break;
  }
}

void launch_pair(int kind, bool st, const BatchInst* inst, const int* o1, int n1, const int* o2, int n2, int parity,
                 cudaStream_t s) {
  if (st)
    launch_pair_t<true>(kind, inst, o1, n1, o2, n2, parity, s);
  else
    launch_pair_t<false>(kind, inst, o1, n1, o2, n2, parity, s);
}

// one launch of the mixed kernel over n items with `grid` blocks (at most n); queue:
// the kernel's two counters, zero before the launch (and after it)
void launch_mixed(int kind, bool st, const BatchInst* inst, const int4* items, int n, int grid, int p1, int p2,
                  unsigned* queue, cudaStream_t s) {
  if (n <= 0) return;
  n *= kParts;
  grid = grid < n ? grid : n;
#define PPLBM_KM(K)                                                                   \
  do {                                                                                \
    if (st)                                                                           \
      k_batch_mixed<K, true><<<grid, kBlock, 0, s>>>(inst, items, n, p1, p2, queue);\
    else                                                                              \
      k_batch_mixed<K, false><<<grid, kBlock, 0, s>>>(inst, items, n, p1, p2, queue);\
  } while (0)
  switch (kind) {
    case kUnitTau: PPLBM_KM(kUnitTau); break;
    case kShearTau: PPLBM_KM(kShearTau); break;
    default: PPLBM_KM(kFullMrt); break;
  }
#undef PPLBM_KM
}

// the collision pass alone, over every instance
void launch_collision_pass(int kind, bool st, const BatchInst* inst, const int* o2, int n2, int parity,
                           cudaStream_t s) {
#define PPLBM_K2(K)                                                                   \
  do {                                                                                \
    if (st)                                                                           \
      launch_dependent(k_batch_collide<K, true>, n2 * kParts, kBlock, s, inst, o2, parity); \
    else                                                                              \
      launch_dependent(k_batch_collide<K, false>, n2 * kParts, kBlock, s, inst, o2, parity); \
  } while (0)
  switch (kind) {
    case kUnitTau: PPLBM_K2(kUnitTau); break;
    case kShearTau: PPLBM_K2(kShearTau); break;
    default: PPLBM_K2(kFullMrt); break;
  }
#undef PPLBM_K2
}

// the density/psi pass alone, over every instance (refreshes psi and the moments)
void launch_density_pass(int kind, const BatchInst* inst, const int* o1, int n1, int parity, cudaStream_t s) {
  switch (kind) {
    case kUnitTau: launch_dependent(k_batch_rho_psi<kUnitTau>, n1 * kParts, kBlock, s, inst, o1, parity); break;
    case kShearTau: launch_dependent(k_batch_rho_psi<kShearTau>, n1 * kParts, kBlock, s, inst, o1, parity); break;
    default: launch_dependent(k_batch_rho_psi<kFullMrt>, n1 * kParts, kBlock, s, inst, o1, parity); break;
  }
}

}  // namespace
}  // namespace pplbm
