// pdl.cuh -- programmatic dependent launch for kernels that follow one another on a stream: the
// next launch's CTAs are scheduled, and compute their indices, while the last CTAs of the current
// one still run.  A kernel launched by launch_pdl calls pdl_enter() before its first global access;
// it returns when every earlier kernel of the stream has completed and its writes are visible, so the
// order of memory accesses is that of ordinary launches.  launch_pdl_if(false, ...) is an ordinary
// launch, for which pdl_enter() does nothing.
//
// Which launches are dependent: an early CTA goes where there is room, and where the running launch leaves
// room on some SMs only, two settle on one of them and the unevenness persists from launch to launch.
// So the FP64 step is dependent behind itself only (its shares are one CTA per SM: 200^2 5.2 us per
// step, 8.0 when it settled behind another kernel), the row pipeline behind a pass of the same depth
// that is on few SMs or fills them, and the FD4 pairs where two launches cannot share the SMs.  The
// one-step streaming kernel (many small CTAs), the register tiles and BGK tiles (an SM's worth of
// registers per CTA) and the transfers always are: behind a transfer, 17 grids, seven repetitions, the
// streaming kernel is 1.01 to 1.6 times as fast as with ordinary launches, the BGK tiles 0.97 to 1.1.
//
// The pointers such a kernel reads through are not __restrict__: that would allow the compiler to read
// them before pdl_enter(), or through the read-only path, whose data may not change while the kernel
// runs -- and it runs while its predecessor writes them.  (The row pipeline, which reads memory by
// cp.async in volatile assembly alone, may keep it.)
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace sslbm {

__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

template <typename... P, typename... A>
cudaError_t launch_pdl_if(bool dependent, void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                          A&&... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}

template <typename... P, typename... A>
cudaError_t launch_pdl(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  return launch_pdl_if(true, kern, grid, block, smem, s, std::forward<A>(args)...);
}

}  // namespace sslbm
