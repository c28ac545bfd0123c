// Launches that overlap the end of the kernel before them (programmatic dependent launch): the
// dependent kernel's CTAs may become resident once every CTA of the one before has begun, and wait
// in wait_for_previous() until it has ended and its writes are visible.  A kernel that is launched
// the ordinary way finds nothing to wait for.  The chain index -> walk -> fix-up of a one-shot
// product saves most of three launch gaps by it (200,003 x 41 banded, FP32: 35.6 -> 30.2 us).
//
// The next kernel's CTAs share their SM with the last CTAs of the one before, and its split between L1
// and shared memory with them.  Kernels that want the same split (the SPLIT chain) let the next
// begin at their start.  The persistent ROWS_TMA does so at its end: begun earlier, its successor
// was placed unevenly (2M x 50 banded 254 -> 290 us, at the end 252; 100^3 27-point 68.4 -> 66.4; 500,001 x 37
// banded, FP32, k = 3, 84.4 -> 81.9).  ROWS and ROWS_DIRECT are launched the ordinary way:
// ROWS_TMA beside the last CTAs of ROWS found little shared memory (a pair of products
// 297 -> 506 us), and ROWS_DIRECT beside those of ROWS_TMA little L1 (332 -> 353).
#pragma once
#include <cuda_runtime.h>

namespace gbs {

// First statement of a kernel that is launched with launch_dependent.
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next launch_dependent kernel begin to take its place once every CTA is here (or gone).
__device__ __forceinline__ void allow_next() { asm volatile("griddepcontrol.launch_dependents;"); }

template <typename... P, typename... A>
cudaError_t launch_dependent(void (*kernel)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t s,
                             A... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace gbs
