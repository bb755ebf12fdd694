// Programmatic dependent launch of the step kernels that a lattice's steps
// chain: step k + 1 is brought up while the blocks of step k finish (launch,
// parameters, index arithmetic, table prefetches) and waits, before its first
// access to a population, until step k has completed and its writes are visible.
// Without it a step costs the launch and its dependency on top of the kernel, in
// units of about 2 us back to back.
//
// A kernel launched so calls pdl_wait in every thread before its first access to
// a population and reads populations with ld_pop: the previous step writes them
// while this kernel is resident, so the read-only path (ld.global.nc) is not for
// them.  The next step is let in after the wait, not before: it then comes up
// beside the running step, and no further ones pile up behind it (let in at the
// start, a dozen waiting steps filled the SMs and a small lattice's step took 66
// or 164 us instead of 16 or 28).  A kernel launched without the attribute (graph
// nodes) finds both instructions empty.
#pragma once

#include <cuda_runtime.h>

namespace rlbm {

__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Coherent loads of populations; volatile, so that they stay behind the wait.
__device__ __forceinline__ float ld_pop(const float* p) { return __ldca(p); }
__device__ __forceinline__ double ld_pop(const double* p) { return __ldca(p); }
__device__ __forceinline__ unsigned short ld_pop(const unsigned short* p) { return __ldca(p); }
__device__ __forceinline__ uint2 ld_pop(const uint2* p) { return __ldca(p); }

template <class... P, class... A>
cudaError_t launch_pdl(void (*kernel)(P...), unsigned grid, unsigned block, cudaStream_t s, A&&... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace rlbm
