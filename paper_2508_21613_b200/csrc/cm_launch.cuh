// Launches that overlap with the end of the kernel before them on the stream (programmatic dependent launch): the blocks
// of the later kernel start as soon as those of the earlier one have all passed after_previous(), and get as far as their
// own after_previous(), which waits until the earlier kernel is complete and its results are visible.  What stands before
// it may only read what no kernel of the sequence writes: the profile, the feasible lists, the descriptor tables.
// (A kernel waits before it lets the next one start, so a block is at most one kernel ahead.)
// One failure of the 256-device job is a chain of twelve launches, one of the 32-device job of five.
#pragma once

#include <utility>

#include <cuda_runtime.h>

namespace cm {

__device__ __forceinline__ void after_previous() {
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
}

template <typename... Params, typename... Args>
inline cudaError_t launch_next(void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, Args &&...args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(std::forward<Args>(args))...);
}

}  // namespace cm
