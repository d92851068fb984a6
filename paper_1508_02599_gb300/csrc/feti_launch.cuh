// Launches that start before their predecessor in the stream has ended
// (programmatic dependent launch).  The kernels of a PCG iteration on small
// decompositions run 2 to 8 us each, of which several are the launch and the
// first instructions: with launch_dep the CTAs of the next kernel are placed
// while the previous one runs, and wait in dep_wait for its end.  dep_go comes
// after dep_wait: with it first, the CTAs of several kernels waited at once and
// a Newton load step took 592 ms instead of 476.
//
// Before dep_wait such a kernel reads only what no kernel of the same
// uninterrupted chain of launches writes (the topology's tables, the R rows and
// the coarse inverse of the setup); it takes its pointers to all other memory
// through fresh() after it: the compiler may otherwise move a load through a
// __restrict__ pointer above the wait.  All its threads wait, so a kernel that
// has ended implies that everything before it has.
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace feti {
namespace {

// Waits until the previous kernel of the stream has ended and its writes are
// visible.
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel's CTAs be placed (once every CTA of this one has said so
// or ended).  Large operators' fixed-point applies (launch_symv_fixed) neither
// say it nor are launched this way: waiting CTAs beside them, or CTAs of theirs
// placed unevenly beside the gather, cost more than the launch.
__device__ __forceinline__ void dep_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename T>
__device__ __forceinline__ T* fresh(T* p) {
  asm volatile("" : "+l"(p)::"memory");
  return p;
}

template <typename... P, typename... A>
cudaError_t launch_dep(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(std::forward<A>(args))...);
}

}  // namespace
}  // namespace feti
