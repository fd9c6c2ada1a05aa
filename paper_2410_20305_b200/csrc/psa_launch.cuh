// Programmatic dependent launch.  A kernel launched with launch_behind(true, ...) may start, with its set-up and its wait
// for a place on an SM, while the kernel before it in the stream still runs.  behind_wait() returns when that kernel has
// completed.  behind_go() lets the next kernel start once all blocks of this one have called it or ended.
// The order of a stream is kept like this: some thread of every kernel launched behind another one calls behind_wait()
// before the kernel can end, and whatever the kernel before it may still read or write is touched only after that.
#pragma once
#include <cuda_runtime.h>


namespace psa {

__device__ __forceinline__ void behind_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void behind_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... Params, typename... Args>
void launch_behind(bool behind, void (*kernel)(Params...), dim3 grid, unsigned block, size_t smem, cudaStream_t stream,
                   Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = behind ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, Params(args)...);
}

}  // namespace psa
