// Dependent launches.  A collection is three short kernels or more in a row (weight image, rollout, advantages) and a gradient
// with its optimiser step five; launched one after the other each pays a launch gap of a few microseconds.  They are launched
// with programmatic serialization instead: a kernel may start while the one before it still runs, does what needs nothing
// from it (barriers, tensor memory, zeroed tiles) and then waits until that one is complete and its writes are visible.
// Rules for a kernel that is launched like this:
//   - Every block waits, whatever it does before: a kernel's completion then implies that of all before it.  All threads of a
//     block wait, but for those that only read what an even earlier kernel is known to have finished (what fetches rows in
//     ppo_net_tc_kernel inside mava_ppo_update; launch_ppo_grad has the argument, which also lets step_image_kernel read the
//     optimiser's state before its wait).
//   - Memory that a kernel in front may still be writing is not constant for the kernel's lifetime, so it must not be declared
//     so: no __restrict__ on its parameters and no load through the non-coherent path (__ldg, ld.global.nc).  Either lets the
//     compiler take a load for an invariant and move it over the wait.  Where loads should go out in a batch they are __ldcg.
//   - A kernel that lets its successor start (dependents_may_start) does so for successors that have room beside it.  The
//     weight-image kernels in front of a rollout do not: blocks that want an SM each and arrive while others still sit on
//     some SMs are doubled up on the rest (8x8 evaluation block 181 -> 192 us).
#pragma once
#include <cuda_runtime.h>

namespace mava {

__device__ __forceinline__ void dependents_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_dependent(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, const A &...args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cfg.attrs = &attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

}  // namespace mava
