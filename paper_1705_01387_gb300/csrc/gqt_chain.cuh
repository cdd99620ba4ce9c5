// gqt_chain.cuh -- launches of the order chains with their start overlapped.
//
// An order of a small or middling system takes 4 to 20 us, and the start of its grid after
// the end of the one before costs 1 to 3 on a plain stream, less in a graph.  The
// kernels of a chain are launched with programmatic stream serialisation: a grid is set
// up while the one before runs out, and waits (chain_wait) until that has ended and its
// results are visible.  A Kubo-Bastin chain of 256 FP64 orders, 18,432 elements: 3.59 ->
// 2.83 ms with its contraction; of 500 FP32 orders, 131,072 elements: 5.83 -> 4.59 ms; rows
// replayed as graphs gain 1 to 5%.  No kernel lets its dependents start before its own
// CTAs end (griddepcontrol.launch_dependents): several grids of waiting CTAs then pile
// up on the SMs, and the same chains take 2.90 and 5.29 ms, those in graphs longer than
// without any overlap.
//
// A kernel launched this way reads before chain_wait only what no kernel of the chain
// writes (the handle's H~ and block tables), and everything else after it by plain
// loads: a read-only load (__ldg, or a const __restrict__ pointer) might be moved up over
// the wait.  The first launch of a chain is an ordinary one, behind whatever prepared
// H~.  Every CTA waits before it ends, so that the end of a grid implies the end of all
// grids before it.
#pragma once

#include <cuda_runtime.h>

#include "gqt_internal.h"

namespace gqt {

__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// kern<<<grid, block, smem, st>>>(args...), overlapped with the launch before if chained.
template <class... P, class... A>
inline void launch_chain(bool chained, void (*kern)(P...), int grid, int block, size_t smem, cudaStream_t st,
                         A&&... args) {
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = chained ? 1 : 0;
  check_cuda(cudaLaunchKernelEx(&cfg, kern, P(args)...), "chain launch");
}

}  // namespace gqt
