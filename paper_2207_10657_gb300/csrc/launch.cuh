// Launches of the spectral passes as a chain: a pass is set up while the one
// before it ends, and waits on the device for that grid (programmatic dependent
// launch).  A product of a small cell is three to five kernels of a few
// microseconds, and the gaps between dependent launches were up to a third of
// its time: products at 512^2 FP32 27.8 -> 21.2 us, 32^2 FP64 34.8 -> 27.2 us,
// 128^3 160 -> 148 us, 256^3 1006 -> 997 us.
//
// The passes do not trigger their dependents early (griddepcontrol.
// launch_dependents): with the trigger at a kernel's start the next grids'
// waiting blocks hold slots and spread the running blocks unevenly (512^2
// 39.5 us, 256^3 1035 us; after the wait 21.7 and 1040 us).
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace rve {

// First statement of every chained kernel: wait until the previous grid has
// finished and its writes are visible.  Nothing is read or written before it.
// A no-op in an ordinary launch.
__device__ __forceinline__ void chain_begin() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch a kernel that starts with chain_begin().  Under stream capture the
// launch is an ordinary one: captured graphs (the CG loop's conditional body
// among them) keep full kernel dependencies.  What programmatic edges would
// give there has not been measured.
template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A&&... args) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusActive;
  if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) {
    cudaGetLastError();  // another stream captures: launch in the ordinary way
    cap = cudaStreamCaptureStatusActive;
  }
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = cap == cudaStreamCaptureStatusNone ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(std::forward<A>(args))...);
}

}  // namespace rve
