// Overlap of one kernel's start with the end of the one before it on the
// stream (programmatic dependent launch).  A kernel launched with
// launch_overlapped may be resident before its predecessor has ended; it calls
// grid_wait() before it touches memory, which returns when the predecessor has
// completed and its writes are visible, and grid_release() after that, which
// lets the next kernel become resident as this one's last blocks drain.  In
// this order no kernel starts before the one two places earlier has ended, so
// a buffer that is read, then rewritten, then read again along a chain of
// updates never meets a reader of its old contents.
// Between short dependent kernels the launch itself took 2 us or more.
#pragma once
#include <cuda_runtime.h>

namespace xlb {

__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
inline cudaError_t launch_overlapped(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                     A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

}  // namespace xlb
