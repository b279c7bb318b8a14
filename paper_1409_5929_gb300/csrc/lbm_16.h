// lbm_16.h -- one time step per launch, boundary nodes included, 16-bit storage in two buffers
// (lbm_16.cu).  The node updates are those of lbm_nodes.cuh, bit for bit what the kernels of
// lbm.cu make of them (checked on states of every geometry; temperatures of the pipe with inlet on
// grids of a few nodes differ by one FP32 rounding).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "../../include/lbm.h"
#include "lbm_physics.cuh"

namespace lbm {

struct Step16 {
    Consts<float> c;
    void *f[2];        // flow planes of the two buffers
    float *g[2];       // temperature planes
    const float* phi;
    int64_t plane;
};

// One step of a problem from buffer `from` to the other, the interior from global loads.
cudaError_t launch16(int storage, const Step16& s, int from, cudaStream_t stream);

// Fields of the state in buffer `which`, as lbm_moments (outputs nr nz floats in device memory or NULL).
cudaError_t launch_fields16(int storage, const Step16& s, int which, float* rho, float* ur, float* uz, float* T,
                            cudaStream_t stream);

// One step of the instances of a batch.  Blocks: (2 instance + kind, first interior pair or boundary
// node), kind 1 for boundary nodes.
struct Blocks16 {
    std::vector<int2> even, odd;   // instances with even and odd nz
};
Blocks16 blocks16(const std::vector<lbm_params>& p, const std::vector<int>& act);
cudaError_t launch_batch16(int storage, const Step16* inst, const int2* blocks, int n, bool odd_nz, int from,
                           cudaStream_t stream);

}  // namespace lbm
