// Kernel launches that overlap their set-up with the end of the launch before (programmatic
// dependent launch).  In a call that overlaps (ProfilerGuard) a kernel launched with launch() may
// start while its predecessor in the stream still runs; it calls pdl_begin() before it touches
// memory that any earlier launch of the stream writes or reads, which lets its own successor start
// likewise and waits until everything before it is done and visible.  What needs only the plan's
// constant tables may come before.  On small meshes the gaps between launches are most of a step:
// run_32p_64g (about 170 launches) 947 -> 563 us.  Which calls do it: small_mesh in api.cu.
#pragma once
#include <cuda_runtime.h>

#include <utility>

#include "profiler.cuh"

namespace cola {

__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// (errors are left for the cudaGetLastError that follows every launch)
template <class... P, class... A>
inline void launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = t_overlap ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(std::forward<A>(args))...);
}

}  // namespace cola
