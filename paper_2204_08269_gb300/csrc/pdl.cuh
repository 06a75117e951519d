// Programmatic dependent launch of the transform's kernel chain: a kernel is put on the SMs while
// the last blocks of its predecessor still run, and blocks in pdl_enter until the predecessor has
// completed and its writes are visible.  That hides the launch latency and the tail of every link
// (a B = 1 step has 18 of them).  Every kernel launched through launch_pdl calls pdl_enter before
// its first access to global memory that is not a constant of the plan; since each link waits for
// the one before it, a kernel sees everything earlier in the stream.
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace jtfs {

// The next kernel may be launched once every block of this grid has called this or exited.
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// Returns when the preceding kernels have completed (at once in a kernel launched normally).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_enter() {
  pdl_trigger();
  pdl_wait();
}

template <typename... Params, typename... Args>
inline void launch_pdl(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem,
                       cudaStream_t st, Args&&... args) {
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);   // errors: cudaGetLastError
}

}  // namespace jtfs
