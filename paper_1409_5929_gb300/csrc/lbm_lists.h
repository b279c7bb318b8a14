// lbm_lists.h -- device copies of the lists (tiles, blocks) that follow the active instances of a batch.
#pragma once
#include <cuda_runtime.h>

#include <stddef.h>

namespace lbm {

struct DeviceList {
    void* dev = nullptr;
    size_t cap = 0;   // bytes
};

struct ListUpload {
    DeviceList* list;
    const void* data;   // host memory, unchanged until the call returns
    size_t bytes;
};

// Replace the contents of n lists, growing those that are too short, and wait.  All or nothing: if an
// allocation fails, every list keeps its memory and its contents, so that launches made with the counts
// of those contents stay in bounds.
inline cudaError_t upload_lists(const ListUpload* u, int n, cudaStream_t stream) {
    constexpr int MOST = 8;
    if (n > MOST) return cudaErrorInvalidValue;
    void* grown[MOST] = {};
    for (int k = 0; k < n; ++k) {
        if (u[k].bytes <= u[k].list->cap) continue;
        const cudaError_t e = cudaMalloc(&grown[k], u[k].bytes);
        if (e == cudaSuccess) continue;
        for (int j = 0; j < k; ++j) cudaFree(grown[j]);
        (void)cudaGetLastError();
        return e;
    }
    for (int k = 0; k < n; ++k) {
        if (!grown[k]) continue;
        cudaFree(u[k].list->dev);
        u[k].list->dev = grown[k];
        u[k].list->cap = u[k].bytes;
    }
    for (int k = 0; k < n; ++k) {
        if (!u[k].bytes) continue;
        const cudaError_t e = cudaMemcpyAsync(u[k].list->dev, u[k].data, u[k].bytes, cudaMemcpyHostToDevice, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaStreamSynchronize(stream);
}

}  // namespace lbm
