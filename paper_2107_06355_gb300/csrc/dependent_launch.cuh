// Programmatic dependent launch of the kernels that follow one another in a stream (the
// passes of a step, of an adjoint step, of a finite-difference step).
//
// The next kernel's blocks become resident while the previous one's last blocks run, so
// its launch costs nothing on the critical path; each kernel waits for the launches before
// it to complete before its first access to memory that a kernel writes, and only
// then lets its own successor start: with the two calls the other way round several
// launches pile up on the SMs, and later ones find their places unevenly (33,700 nodes,
// two-phase: 14.5 us per step against 10.0). Single lattice, us per step without / with:
// 20,000 nodes 12.4 / 8.4, 150,000 nodes 20.1 / 15.2, 1.05 M nodes 60.8 / 55.7; two-phase
// 33,700 nodes 14.1 / 10.0, 1.05 M 73.8 / 68.4.
#pragma once

#include <cuda_runtime.h>

namespace pplbm {

// A grid of cols x rows tiles, the rows beyond the y axis' 65,535 blocks on the z axis (the
// last layer may be partly empty), and a block's tile row in it.
inline dim3 tile_grid(int cols, int rows) {
  const int layer = rows < 65535 ? rows : 65535;
  return dim3((unsigned)cols, (unsigned)layer, (unsigned)((rows + layer - 1) / layer));
}
__device__ __forceinline__ int tile_row() { return (int)(blockIdx.z * gridDim.y + blockIdx.y); }

// at the start of a kernel launched by launch_dependent, before any access to memory that a
// kernel writes
__device__ __forceinline__ void begin_dependent() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
}

template <class... Params, class... Args>
cudaError_t launch_dependent(void (*kernel)(Params...), dim3 grid, dim3 block, cudaStream_t s, const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

}  // namespace pplbm
