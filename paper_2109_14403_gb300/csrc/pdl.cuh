// pdl.cuh -- chains of small dependent kernels: programmatic dependent launch.
//
// A kernel launched by launch_chained may be set up while the one before it in
// the stream still runs (its CTAs take what room is left once all of the
// predecessor's have started), and waits inside for that one to complete with
// its writes visible.  Hides some 2 us of launch and drain per kernel, which
// is much of a kernel here (a training step of 32 samples is 12 of them).
// Rules: every kernel of a chain calls chain_begin() first, before it reads or
// writes any memory; so each completes only after the whole chain before it,
// and a kernel of any other kind before or after the chain is ordered as usual.
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace dmn {

__device__ __forceinline__ void chain_begin() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The result of a launch; a failed one is taken off the thread's error state too,
// as cudaGetLastError after <<<>>> does: it has been reported, and left there it
// would be found by the next launch check, the caller's own included.
inline cudaError_t launch_status(cudaError_t e) {
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

// overlap = false: an ordinary launch of such a kernel
template <typename... P, typename... A>
cudaError_t launch_chained(bool overlap, void (*f)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                           A &&...args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = overlap ? 1 : 0;
  return launch_status(cudaLaunchKernelEx(&cfg, f, P(std::forward<A>(args))...));
}

}  // namespace dmn
