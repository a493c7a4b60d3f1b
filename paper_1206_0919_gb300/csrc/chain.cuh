// chain.cuh -- back-to-back sweeps of one stream overlapped at their ends.
//
// A sweep reads what the one before it wrote, so it cannot start early, but
// its launch can: the blocks of the next sweep are put on the SMs as those of
// the previous one leave them and wait there, instead of the launch beginning
// when the last block has ended.  Worth it for single launches (64^3, a step
// and its totals per call: 53 -> 49 us a call); inside a graph the edges are
// already short and it loses (48^3, 90 sweeps: 436 -> 463 us), and the
// streaming sweeps, whose work shares follow the order in which blocks come to
// an SM, lose too (200^3: 23.1 -> 23.5 ms).
#pragma once

#include <cuda_runtime.h>

namespace shasta {

// First thing in a chained kernel, before any access to the state: lets the
// next launch begin once every block of this one has started, and waits for
// the previous kernel of the stream to have ended with its writes visible (at
// once where the launch is not chained).
__device__ __forceinline__ void chain_begin() {
#if __CUDA_ARCH__ >= 900
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
#endif
}

// chain: overlapped as above, for kernels that call chain_begin.
inline cudaError_t launch_sweep_kernel(const void* fun, dim3 grid, dim3 block, void** args, size_t smem, bool chain,
                                       cudaStream_t s) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = chain ? 1 : 0;
  return cudaLaunchKernelExC(&cfg, fun, args);
}

}  // namespace shasta
