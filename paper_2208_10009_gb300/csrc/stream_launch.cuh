// stream_launch.cuh -- launches of the pipeline's kernels with programmatic stream serialisation:
// a kernel's launch is processed while its predecessor's last blocks run, and its blocks wait for
// the predecessor's completion (and its memory) in wait_predecessor, the first statement of every
// kernel launched this way.  All blocks wait, also those that then find nothing to do, so the
// order is transitive along the stream.  No kernel lets its successor in before its blocks exit
// (griddepcontrol.launch_dependents): the waiting blocks then hold slots and poll beside it
// (60 FP64 iterations of 4,026 paths 700 -> 790 us, the office call 6.22 -> 6.53 ms).  A launch and
// refinement is eight kernels, most of them a few microseconds long when paths are few; with the
// memsets and the transmitter copy gone into them: a room's call 256 -> 219 us, the clutter's 342
// -> 314, the canyon's 1219 -> 1181.
#pragma once

#include <cuda_runtime.h>

namespace sbr {

__device__ __forceinline__ void wait_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t s, const A &...args) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace sbr
