// Launches of the time step's kernels.  In the chained form (Geom::chain) they
// use programmatic dependent launch: a kernel may be placed on the SMs, and
// run up to its chain_wait(), while the kernel before it in the stream (or
// captured graph) still runs; chain_wait() returns when that kernel has
// completed and its writes are visible.  It hides the launch latency and the
// start of the blocks between the steps, which small lattices spend most of
// their time on (4x49x49 FP64, two kernels per step: 10.3 -> 9.6 us per step,
// 8.1 us with the longer graphs of long_chunk_len).  Lattices of many short
// blocks are launched plainly: the wait costs every block, and the plain
// loads it requires are slower in register-bound kernels (512x256x256 FP16 AA
// step: 4 % slower chained).
//
// Every kernel launched chained calls chain_wait() in every thread before it
// touches memory that other kernels write, so each kernel completes after all
// its predecessors; it also lets the next one be placed.  The kernels
// read such memory by plain loads (the read-only path may be served from lines
// cached before the wait).
#pragma once

#include <cuda_runtime.h>

namespace lbm {

__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... P, typename... A>
inline cudaError_t chain_launch(int chain, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                A&&... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &at;
  c.numAttrs = chain ? 1 : 0;
  return cudaLaunchKernelEx(&c, kernel, P(args)...);
}

}  // namespace lbm
