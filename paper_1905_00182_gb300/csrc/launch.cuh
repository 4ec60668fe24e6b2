// launch.cuh -- launches of a stage's kernels: a kernel's launch overlaps the end of the one before
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace ibfsa {

// First statement of every kernel that launch() starts: waits until the kernels before it in the
// stream are complete and their writes visible.
__device__ __forceinline__ void begin_kernel() { cudaGridDependencySynchronize(); }

// A stage of a small grid is 7 to 10 kernels of 8 to 70 us, and an ordinary launch begins after the
// previous kernel's memory flush: ~2 us a kernel.  Programmatic serialization has the next kernel's
// blocks set up by then, waiting in begin_kernel.  No kernel lets its successor in early
// (cudaTriggerProgrammaticLaunchCompletion): its blocks then crowd onto the SMs that run out first,
// and a pass of one to two blocks per SM takes up to twice its time.  Times of whole cases with
// ordinary launches / these / an early trigger in every kernel: 256^2 FP64 WENO5, 10 steps 5.35 /
// 4.89 / 7.16 ms; 99 x 77 x 85 FP32, 4 steps 1.85 / 1.69 / 1.89; 1021 x 771 FP32 with
// characteristic faces, 6 steps 1.97 / 1.71 / 1.82; 512^3 FP32, 2 steps 72.9 / 72.2 / 74.1.
// Errors are left to cudaGetLastError, as after <<<>>>.
template <typename... P, typename... A>
inline void launch(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t st,
                   A &&...args) {
  cudaLaunchAttribute serial{};
  serial.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  serial.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &serial;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

}  // namespace ibfsa
