// lbm_dependent.h -- launch of a kernel that may start while the one before it still runs.
#pragma once
#include <cuda_runtime.h>

// Launch with programmatic dependent launch: the kernel's blocks may start while the launch before
// it still runs and wait for its end (griddepcontrol.wait) before their first access to memory.
// What earlier launches write is read behind that wait by ordinary loads: the read-only ones (__ldg,
// const __restrict__ kernel parameters) are for data that stays unchanged from the kernel's start.
template <class K, class... Args>
cudaError_t launch_dependent(K kernel, unsigned blocks, unsigned threads, size_t shared, cudaStream_t stream,
                                    Args... args) {
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = shared;
    cfg.stream = stream;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}
