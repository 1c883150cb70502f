// Chained launches: a kernel is launched while its predecessor in the stream still runs.
//
// A solve is a chain of launches of 5 to 100 us, each of which used to wait for the last block of the one before
// it and then for the launch itself, about 1 us a launch.  launch_chained() launches with programmatic stream
// serialisation; the kernel calls chain_wait() before it reads or writes anything that another launch touches:
// it returns when the previous launch has completed and its writes are visible.  Every block of a chained kernel
// calls it (also those with nothing to do), so a launch never completes before its predecessor, and a launch that
// is not chained keeps the stream's usual order.  In a captured stream the launches are ordinary ones.
//
// A kernel's blocks come in as the last blocks of its predecessor leave; but for the MMA kernel behind its gather
// (chain_next) they are not let in earlier: blocks that wait on an SM take the place of working ones where a kernel
// counts on an even spread over the SMs.  Subdomain inverses of 30x30x13 cells: 228 ms with ordinary launches,
// 226 ms so, 349 ms let in early; its gradient evaluation 14.1, 13.4 and 13.8 ms; sphere 12^3 solve 1.91, 1.61 and
// 1.64 ms; 16 sparse subdomains 17.6, 15.9 and 16.7 ms; training epochs at 2048 inputs 16.2, 14.1 and 17.0 ms.
#pragma once
#include <cuda_runtime.h>

namespace mwk {

__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Lets the next launch's blocks in before this launch ends (the one use: the gather lets the MMA kernel in, whose
// blocks then set up and start copies that do not depend on the gather).
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
inline void launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(s, &st);
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = st == cudaStreamCaptureStatusNone ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace mwk
