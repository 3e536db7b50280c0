// The two step kernels of the pseudopotential D2Q9 lattice Boltzmann method for
// one lattice, and their helpers (sm_103a, FP64). The per-node arithmetic is in
// step_device.cuh.
//
// K1 rho_psi : reads the 9 pre-collision populations of a node (coalesced SoA),
//              forms the moments the collision needs (rho = sum f, Eq. Density;
//              j = sum f c; plus the stress moments when they relax), evaluates the
//              equation of state and psi (Eq. InteractionPotential), writes psi and
//              the moments.
// K2 collide : reads the node's psi stencil (periodic wrap in x, periodic or wall
//              ghost rows in y), computes the Shan-Chen force
//              (Eq. ShanChenForce), the velocity with the F/2 shift (Eq. Momentum),
//              the MRT collision with the Li source (Eqs. OperatorMRT, LiFS,
//              GFS), optionally the surface-tension source of Sec. V's
//              technique, and pushes f* to the neighbours (streaming, Eq. LBE),
//              with half-way bounce-back at walls (Sec. IV).
#include <cuda_runtime.h>

#include "cluster_steps.cuh"
#include "dependent_launch.cuh"
#include "step_device.cuh"

namespace pplbm {

namespace {

// K2's tile, one warp along x, and K1's block of as many nodes. Small blocks spread a small
// lattice evenly: with 8 warps per block 33,700 nodes are 153 blocks for 152 SMs (two-phase
// step 16.9 us, 14.5 with 2 warps); large lattices run at the same rate either way.
constexpr int kTX = 32, kTY = 2, kStepThreads = kTX * kTY;

template <int KIND>
__global__ void __launch_bounds__(kStepThreads) k_rho_psi(const __grid_constant__ StepArgs a) {
  begin_dependent();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;  // n < 2^31 / 9
  if (i >= (int)a.n) return;
  rho_psi_node<KIND>(a, a.f_in, i);
}

// 40 resident warps per SM (48 registers) except the two-phase kernel with the
// surface-tension source (32 warps, 64 registers), which would spill too much
constexpr int collide_blocks(int kind, bool st) { return ((st && kind == kShearTau) ? 32 : 40) / kTY; }

template <int KIND, bool FIELDS, bool ST = false>
__global__ void __launch_bounds__(kStepThreads, collide_blocks(KIND, ST)) k_collide(const __grid_constant__ StepArgs a, double* rho_o, double* ux_o,
                                                                                     double* uy_o, double* psi_o) {
  begin_dependent();
  const int x = blockIdx.x * kTX + threadIdx.x, y = tile_row() * kTY + threadIdx.y;
  if (x >= a.nx || y >= a.ny) return;
  collide_node<KIND, FIELDS, ST>(a, x, y, rho_o, ux_o, uy_o, psi_o);
}

// f_i = f_i^eq(rho0, u0), Eq. EquilibriumDistribution (c_s^2 = 1/3). Bound by the FP64 pipe:
// with c.u and the polynomial formed per population (63 FP64 instructions per node) 12.9 M
// nodes took 1.54 ms; 0.91 with what the directions of a line share formed once (33), and
// 0.18 at rest (3).
__global__ void k_init_eq(int64_t n, double* f, const double* rho0, const double* ux0, const double* uy0,
                          int* err) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double rho = rho0[i];
  if (!(rho > 0.0 && rho < 1e300)) atomicOr(err, 1);
  const double r0 = 4.0 / 9 * rho, r1 = 1.0 / 9 * rho, r5 = 1.0 / 36 * rho;
  if (!ux0 && !uy0) {  // at rest: f_i = w_i rho
    f[i] = r0;
#pragma unroll
    for (int k = 1; k < 9; ++k) f[k * n + i] = k < 5 ? r1 : r5;
    return;
  }
  const double ux = ux0 ? ux0[i] : 0.0, uy = uy0 ? uy0[i] : 0.0;
  // w_i rho (1 + 3 c.u + 4.5 (c.u)^2 - 1.5 u^2): the two directions of a line share the even part
  const double a = fma(-1.5 * ux, ux, fma(-1.5 * uy, uy, 1.0));
  auto line = [&](double cu, double r, int k, int opp) {
    const double even = fma(4.5 * cu, cu, a);
    f[k * n + i] = r * fma(3.0, cu, even);
    f[opp * n + i] = r * fma(-3.0, cu, even);
  };
  f[i] = r0 * a;
  line(ux, r1, 1, 3);
  line(uy, r1, 2, 4);
  line(ux + uy, r5, 5, 7);
  line(uy - ux, r5, 6, 8);
}

// guard: a density pass over the current state, then per-block partials of the
// guard terms (guard_node) over a fixed grid-stride partition, then one block
// reduces them in a fixed order: deterministic
constexpr int kGuardBlocks = 304;
constexpr int kGuardThreads = 256;

__global__ void __launch_bounds__(kGuardThreads) k_guard_partial(const StepArgs a, double* snap, int snap_valid,
                                                                 double* partials) {
  __shared__ double s[kGuardQ][kGuardThreads];
  double v[kGuardQ] = {0.0, 0.0, 0.0, 0.0};
  for (int64_t i = blockIdx.x * (int64_t)kGuardThreads + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * kGuardThreads)
    guard_node(a, i, snap, snap_valid != 0, v);
  guard_block_reduce<kGuardThreads>(v, s);
  if (threadIdx.x < kGuardQ) partials[kGuardQ * blockIdx.x + threadIdx.x] = s[threadIdx.x][0];
}

__global__ void __launch_bounds__(kGuardThreads) k_guard_final(const double* partials, int nblocks, int snap_valid,
                                                               double* out) {
  __shared__ double s[kGuardQ][kGuardThreads];
  double v[kGuardQ] = {0.0, 0.0, 0.0, 0.0};
  for (int k = threadIdx.x; k < nblocks; k += kGuardThreads) {
    v[0] += partials[kGuardQ * k];
    v[1] = fmax(v[1], partials[kGuardQ * k + 1]);
    v[2] += partials[kGuardQ * k + 2];
    v[3] += partials[kGuardQ * k + 3];
  }
  guard_block_reduce<kGuardThreads>(v, s);
  if (threadIdx.x == 0) {
    out[0] = s[0][0];
    out[1] = s[1][0];
    out[2] = s[2][0];
    out[3] = snap_valid ? s[3][0] / s[0][0] : -1.0;
  }
}

template <int KIND, bool ST>
__global__ void __launch_bounds__(kClusterThreads) k_cluster_steps(const __grid_constant__ StepArgs a, int nsteps) {
  __shared__ StepArgs sa[2];
  if (threadIdx.x == 0) {
    sa[0] = a;
    sa[1] = a;
    sa[1].f_in = a.f_out;
    sa[1].f_out = const_cast<double*>(a.f_in);
  }
  __syncthreads();
  cluster_steps<KIND, ST>(sa, 0, nsteps);
}

const void* cluster_kernel(int kind, bool st) {
  switch (kind) {
    case kUnitTau: return st ? (const void*)k_cluster_steps<kUnitTau, true> : (const void*)k_cluster_steps<kUnitTau, false>;
    case kShearTau:
      return st ? (const void*)k_cluster_steps<kShearTau, true> : (const void*)k_cluster_steps<kShearTau, false>;
    default: return st ? (const void*)k_cluster_steps<kFullMrt, true> : (const void*)k_cluster_steps<kFullMrt, false>;
  }
}

dim3 collide_grid(const StepArgs& a) { return tile_grid((a.nx + kTX - 1) / kTX, (a.ny + kTY - 1) / kTY); }

}  // namespace

void launch_rho_psi(const StepArgs& a, void* stream) {
  const unsigned blocks = (unsigned)((a.n + kStepThreads - 1) / kStepThreads);
  cudaStream_t s = (cudaStream_t)stream;
  switch (a.kind) {
    case kUnitTau: launch_dependent(k_rho_psi<kUnitTau>, blocks, kStepThreads, s, a); break;
    case kShearTau: launch_dependent(k_rho_psi<kShearTau>, blocks, kStepThreads, s, a); break;
    default: launch_dependent(k_rho_psi<kFullMrt>, blocks, kStepThreads, s, a); break;
  }
}

void launch_collide(const StepArgs& a, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  const dim3 block(kTX, kTY);
  double* const none = nullptr;
  if (a.kappa_q != 0.0) {  // with the surface-tension source
    switch (a.kind) {
      case kUnitTau: launch_dependent(k_collide<kUnitTau, false, true>, collide_grid(a), block, s, a, none, none, none, none); break;
      case kShearTau: launch_dependent(k_collide<kShearTau, false, true>, collide_grid(a), block, s, a, none, none, none, none); break;
      default: launch_dependent(k_collide<kFullMrt, false, true>, collide_grid(a), block, s, a, none, none, none, none); break;
    }
    return;
  }
  switch (a.kind) {
    case kUnitTau: launch_dependent(k_collide<kUnitTau, false>, collide_grid(a), block, s, a, none, none, none, none); break;
    case kShearTau: launch_dependent(k_collide<kShearTau, false>, collide_grid(a), block, s, a, none, none, none, none); break;
    default: launch_dependent(k_collide<kFullMrt, false>, collide_grid(a), block, s, a, none, none, none, none); break;
  }
}

ClusterShape small_lattice_shape(const StepArgs& a) {
  return cluster_shape(cluster_kernel(a.kind, a.kappa_q != 0.0), kClusterNodes, a.n, a.n, 1);
}

void launch_cluster_steps(const StepArgs& a, ClusterShape shape, int nsteps, void* stream) {
  void* args[] = {(void*)&a, (void*)&nsteps};
  launch_clusters(cluster_kernel(a.kind, a.kappa_q != 0.0), 1, shape, args, (cudaStream_t)stream);
}

void launch_fields(const StepArgs& a, double* rho, double* ux, double* uy, double* psi_out, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  const dim3 block(kTX, kTY);
  switch (a.kind) {
    case kUnitTau: launch_dependent(k_collide<kUnitTau, true>, collide_grid(a), block, s, a, rho, ux, uy, psi_out); break;
    case kShearTau: launch_dependent(k_collide<kShearTau, true>, collide_grid(a), block, s, a, rho, ux, uy, psi_out); break;
    default: launch_dependent(k_collide<kFullMrt, true>, collide_grid(a), block, s, a, rho, ux, uy, psi_out); break;
  }
}

void launch_init_eq(const StepArgs& a, double* f, const double* rho0, const double* ux0, const double* uy0,
                    void* stream) {
  const unsigned blocks = (unsigned)((a.n + 255) / 256);
  k_init_eq<<<blocks, 256, 0, (cudaStream_t)stream>>>(a.n, f, rho0, ux0, uy0, a.err);
}

int guard_blocks() { return kGuardBlocks; }

void launch_guard(const StepArgs& a, double* snap, int snap_valid, double* partials, double* out, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  launch_rho_psi(a, stream);
  k_guard_partial<<<kGuardBlocks, kGuardThreads, 0, s>>>(a, snap, snap_valid, partials);
  k_guard_final<<<1, kGuardThreads, 0, s>>>(partials, kGuardBlocks, snap_valid, out);
}

}  // namespace pplbm
