// Programmatic dependent launch.  A kernel launched with launch_behind(true, ...) may start, with its set-up and its wait
// for a place on an SM, while the kernel before it in the stream still runs.  behind_wait() returns when that kernel has
// completed.  behind_go() lets the next kernel start once all blocks of this one have called it or ended.
// The order of a stream is kept by three rules:
// 1. Some thread of every kernel launched behind another one calls behind_wait() before the kernel can end.
// 2. Whatever the kernel before it may still read or write is touched only after behind_wait(), and is not declared
//    `const T* __restrict__`: that says that nobody writes there while the kernel runs, and the compiler may load it early.
// 3. A kernel that touches anything of others before its behind_wait() (dpo_logp_kernel the logits and labels,
//    psa_bwd_kernel the plan and the tiles of Q, K, V, dO) is launched behind one that calls behind_wait() ahead of
//    behind_go(): all that came before is complete by then.  psa_bwd_kernel calls behind_go() first, so only kernels that
//    wait before they read (psa_fwd_kernel, psa_bwd_delta_kernel, psa_bwd_convert_kernel and those of the loss) may follow it.
#pragma once
#include <cuda_runtime.h>

#include <utility>

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
  cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);   // (converts as a launch with <<<>>> does)
}

}  // namespace psa
