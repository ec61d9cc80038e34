// Launches that may start before the kernel ahead of them in the stream has finished
// (programmatic dependent launch).  Such a kernel sets itself up and then waits, before it
// touches any global memory, until the kernels ahead of it have completed and their writes
// are visible; a kernel lets its successor start early once its own blocks have passed that wait.
// Between the small kernels of a sweep this hides most of the launch latency (all amplitudes of
// 4x4x(1+16+1), 21 calls: 155 -> 122 us).  Letting the successor start before the wait hides no more
// of it, and all kernels of a chain become resident at once: their waiting blocks take the free
// slots, and a grid of fewer blocks than SMs ends up with two on some (852 columns of K = 1024, N = 512
// in 64 x 64 tiles, 112 blocks: 184 us, against 106).
// Such a kernel declares what an earlier one may write without __restrict__ and reads it with
// plain loads: loads that the compiler takes for invariant may move above the wait.  The plan's
// tables keep __restrict__: a copy ahead of a call's first kernel has written them.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace qfx {

// Device: returns when every kernel ahead in the stream has completed (at once in a kernel
// launched the ordinary way).
__device__ __forceinline__ void launch_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Device: the next kernel may start once every block has come here (or ended).
__device__ __forceinline__ void launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Host: launches `kernel`, which calls launch_wait() before its first access to memory that an
// earlier kernel may write, read or still be using.
template <typename... P, typename... A>
cudaError_t launch_early(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(std::forward<A>(args))...);
}

}  // namespace qfx
