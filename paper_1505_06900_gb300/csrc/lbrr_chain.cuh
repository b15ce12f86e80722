// Kernels of a chain: each is launched while the one before it in the stream
// still runs (programmatic stream serialization), prepares what does not depend
// on earlier work, and passes chain_wait() before it touches anything that
// does. The wait returns when the work before is complete and visible; only
// then is the next kernel of the chain let in, so that completion carries along
// the chain. Data read after the wait is read with ordinary loads or
// asynchronous copies, not as read-only for the length of the kernel (no
// const __restrict__ parameters for it). Launch and start-up of a short kernel
// then cost nothing: 50 D2Q9 updates of 128^2 cells and their read-back 61.5 ->
// 48.1 us (50.2 as the runs are now), a training step of 8192 rows 18.5 -> 13.9, a
// closure step of 64^3 38.6 -> 33.9.
#pragma once

#include <cuda_runtime.h>

namespace lbrr {

#ifdef __CUDACC__
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
#endif

template <typename... P, typename... A>
cudaError_t launch_chained(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                           A... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

}  // namespace lbrr
