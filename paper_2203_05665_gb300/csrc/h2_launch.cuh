// Launches of the product's kernels with programmatic dependent launch: a
// kernel's CTAs may be set up while the previous kernel drains; it waits for that
// kernel's completion (and its writes) in pdl_wait before it touches anything
// a product computes.  Every kernel launched through pdl() calls pdl_wait in
// every CTA that does any work, so that a kernel's completion implies that of
// all kernels before it (one launched without it waits for all of them anyway).  A product is a chain of 15 to 30 kernels of a few
// microseconds each around one or two long ones.  Replayed products without and
// with it: 5,120 triangles, one column 70 -> 62 us; ellipsoid of 81,920, order 4,
// one column 726 -> 705 us; 81,920, order 3, 32 columns 903 -> 891 us; batch of six
// 434 -> 412 us; without the early start (pdl_go) 66, 728, 918 and 431 us.
#pragma once

#include <cuda_runtime.h>

namespace h2 {
namespace {

// the next kernel of the stream may be set up from now on
__device__ __forceinline__ void pdl_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// the previous kernel of the stream is complete and its writes are visible
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
inline void pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);   // errors: cudaGetLastError at the end of the product
}

}  // namespace
}  // namespace h2
