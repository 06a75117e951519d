// Programmatic dependent launch of the transform's kernel chain: a kernel is put on the SMs while
// the last blocks of its predecessor still run.  That hides the launch latency and the tail of
// every link (a B = 1 step has 18 of them).  Every kernel launched through launch_pdl waits, on
// every way out, until its predecessor has completed, so that its own completion means that
// everything before it in the stream has completed.  They enter in one of three ways, before the
// first access to global memory that is not a constant of the plan:
//  - pdl_enter, nearly all: the dependents are let go, then the predecessor's end is awaited.
//  - pdl_enter_early: the kernel reads no result of its predecessor, only what was complete before
//    that one let it go; it works beside the predecessor's tail and calls pdl_wait at its end.
//    k_s0 (reads the call's input) and the contraction forms launched `late` (pdl_enter_form; they
//    read Y, and G1 or the weights, as the form before them does).
//  - pdl_enter_ordered: the wait comes before the dependents are let go.  A kernel after which an
//    early one starts, directly or through kernels that let their dependents go at once, has to
//    enter so: k_xfft_sub, the first transform kernel of every call, for k_s0 (the call's input is
//    then complete), and the first form of a contraction stage for the later ones (Y and G1 are).
// griddepcontrol.wait promises visibility to the grid that executes it.  An early kernel takes over
// what the ordered one before it was promised: the writers are complete and their results in global
// memory when that one triggers, and the early grid starts after the trigger.  Its loads must not
// find older lines in an L1: k_s0 reads past it (__ldcg), the contraction forms through TMA (their
// other loads are constants of the plan).
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
__device__ __forceinline__ void pdl_enter_ordered() {
  pdl_wait();
  pdl_trigger();
}
__device__ __forceinline__ void pdl_enter_early() { pdl_trigger(); }   // pdl_wait at its end
// A form of a contraction stage: the first one, or a later one (late), which is independent of it,
// starts on the SMs that it leaves and calls pdl_wait at its end.
__device__ __forceinline__ void pdl_enter_form(int late) {
  if (!late) pdl_wait();
  pdl_trigger();
}

template <typename... Params, typename... Args>
inline void launch_chain(bool early, void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem,
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
  cfg.numAttrs = early ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);   // errors: cudaGetLastError
}

template <typename... Params, typename... Args>
inline void launch_pdl(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem,
                       cudaStream_t st, Args&&... args) {
  launch_chain(true, kernel, grid, block, smem, st, std::forward<Args>(args)...);
}

// The same, not before the predecessor has completed: for kernels of few and long blocks that fit
// an SM several at a time.  Put on the SMs early they gather on those that the predecessor leaves
// first.  The CUDA-core joint kernels, plain FP32, N = 2^16, n1 = 167, 32 frames, B = 1: forward
// 30.5 ms so, 52.0 through launch_pdl.
template <typename... Params, typename... Args>
inline void launch_spread(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem,
                          cudaStream_t st, Args&&... args) {
  launch_chain(false, kernel, grid, block, smem, st, std::forward<Args>(args)...);
}

}  // namespace jtfs
