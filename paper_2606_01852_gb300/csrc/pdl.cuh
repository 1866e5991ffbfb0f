// Programmatic dependent launches: a step's kernel is set up while the step before it still runs.
//
// A path is tens to hundreds of launches of a few microseconds each, one after another; between two
// lie the launch and, in the tensor-core kernels, barriers, tensor maps and TMEM. A kernel launched
// by launch_pdl may start early: it calls pdl_wait before its first access to memory that any
// earlier kernel writes or reads, and pdl_next after it (and after it has its TMEM, so that a later
// kernel never holds what an earlier one still waits for). Each kernel waits for the one before
// it, so the last one's completion is everybody's. The first launch of a call is an ordinary one.
// Such a kernel reads what other kernels write by ordinary loads, L2 loads or TMA, never by the
// read-only path (__ldg, __restrict__): its lines and the compiler may be older than the wait.
// Measured (GB300): one amplitude of a 12-qubit circuit (3 launches) 28.7 -> 24.1 us, 16 amplitudes
// of a 20-qubit one (20 launches) 255 -> 212 us, a 20 x 20 spin glass 12.02 -> 11.81 ms; a 4 x 4
// kicked Ising model replayed from a graph (109 launches) 0.93 ms with and without.
#pragma once

#include <utility>

#include <cuda_runtime.h>

namespace tn {

// The kernels before this one are complete and their writes visible.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// The next kernel may start (it waits for this one's completion by itself).
__device__ __forceinline__ void pdl_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

}  // namespace tn
