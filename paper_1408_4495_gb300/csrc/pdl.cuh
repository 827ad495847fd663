// Programmatic dependent launches: a kernel whose launch may start while the one before it in the
// stream still runs.  Its CTAs take the SMs as the earlier ones leave, set up what needs no data of
// the chain (barriers, tensor memory, index arithmetic, tables that no kernel writes) and then wait.
// Rules that keep a chain of them in order:
//   - a kernel launched with launch_pdl executes pdl_wait (which returns when the grid before it has
//     completed and its writes are visible) in every thread, before it touches anything that a
//     launch of the chain writes, and triggers only after that: so at most two launches of a chain
//     overlap, and the one that runs ahead has only its waiting CTAs on the SMs;
//   - data that an earlier launch of the chain writes is not read through the read-only path (no
//     __ldg, no const __restrict__): such loads may be moved above the wait.  Where that path pays
//     (stencils, plane-wave phases), the kernel is launched plainly and only triggers;
//   - the first kernel of an operator apply is launched plainly: the tables it and the later passes
//     read ahead of their waits were written before it started.
// The instructions do nothing in a plain launch.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

namespace ls {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
// The streaming kernels (FFT passes, stencils, Krylov vectors) let the next launch in early only when
// they have at most one CTA per SM.  There the launch is a good part of the chain: solves of the 2-D
// n = 64 mixed problem with 3 right-hand sides 0.855 -> 0.785 ms, n = 128 with 4 0.839 -> 0.807, n = 32
// FP64 with 1 1.090 -> 1.057, 3-D n = 16 with 4 0.632 -> 0.595.  In larger grids the next kernel's CTAs
// settle on the SMs that empty first and stay unevenly spread: with the trigger in every grid n = 256
// with 16 took 1.757 ms and n = 1024 with 4 8.36 (1.740 and 8.21 without, 1.730 and 8.17 with this
// limit; limits of 304 to 1216 CTAs lie between).
constexpr unsigned PDL_MAX_CTAS = 152;
__device__ __forceinline__ void pdl_trigger_small() {
  if (gridDim.x * gridDim.y * gridDim.z <= PDL_MAX_CTAS) pdl_trigger();
}
__device__ __forceinline__ void pdl_enter() {
  pdl_wait();
  pdl_trigger_small();
}

// launch as a programmatic dependent of the previous kernel in the stream
template <typename... KArgs, typename... Args>
void launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  LS_CUDA(cudaLaunchKernelEx(&cfg, kern, args...));
}

}  // namespace ls
