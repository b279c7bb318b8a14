// lbm_f32.h -- launches of one or more time steps, boundary nodes included, FP32 storage in two
// buffers (lbm_f32.cu; the kernels are in lbm_step32.cuh, lbm_two.cuh and lbm_tile.cuh).  A translation unit of its own:
// how the compiler fuses the multiply-adds of the kernels in lbm.cu shifts with what else is
// compiled beside them, and 16-bit results hang on that bit by bit.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "../../include/lbm.h"
#include "lbm_physics.cuh"

namespace lbm {

// One FP32 state buffer: nine flow planes, five temperature planes.
struct State32 {
    float* f;
    float* g;
};

// The lattice constants with the combinations collide_two works on.
struct Consts32 : Consts<float> {
    // s_e / 36, s_e / 12 and h_e / 6 (s_eps = s_e), s_j / 6 and h_j / 6, s_q / 12 and h_q / 12,
    // s_nu / 4, h_nu / 2 and h_nu / 4
    float a_e, g_u, g_f, a_j, b_j, a_q, b_q, a_nu, b7, b8;
};

// Marches of k_two.  One with boundary nodes takes about 1.6 times as long per row, so those get fewer rows.
struct TwoPlan {
    int strips, first, last;   // strips of columns; rows first .. last are pulled by second steps
    int rows, erows;           // rows of a march without and with boundary nodes
    __host__ __device__ int ends() const { return min(strips, 2); }
    __host__ __device__ int inner() const { return strips - ends(); }
    // end strips: all rows in chunks of erows; inner strips: the first and the last erows rows,
    // and between them chunks of rows
    __host__ __device__ int echunks() const { return (last - first + erows) / erows; }
    __host__ __device__ int outer() const { return min(echunks(), 2); }
    __host__ __device__ int mid() const { return max(last - first + 1 - 2 * erows, 0); }
    __host__ __device__ int chunks() const { return (mid() + rows - 1) / rows; }
    __host__ __device__ int walls() const { return 1 + first; }   // wall rows: 0 too unless it is a pipe axis
    __host__ __device__ int n_wall() const { return strips * walls() + ends() * echunks() + inner() * outer(); }
    __host__ __device__ int n_bulk() const { return inner() * chunks(); }
};

// Tiles of k_tile.
struct TilePlan {
    int T;             // most steps of a launch (the halo); 0: the kernel does not serve this problem
    int cr, cz;        // tile
    int threads;
    int tiles_z, blocks;
    size_t shared;     // bytes of the largest region: 2 x 14 populations, reference, porosity
};

struct Plan32 {
    TwoPlan two;       // strips = 0: the problem is not served
    TilePlan tile;
    bool single;       // one step per launch
};

Consts32 consts32(const Consts<double>& d, const Consts<float>& f);
// What serves a problem (two buffers, 14 planes within 32-bit indices, no discrete heater) on a
// device of `sms` multiprocessors.
cudaError_t plan32(const lbm_params& p, int sms, Plan32* out);
// Steps the next launch takes when `left` remain.  The last launch of a run takes a single step: it
// leaves the previous state in the other buffer.
int steps32(const Plan32& w, int64_t left);
// Launches that n steps take (as many as steps, or fewer if the first one takes more than one).
int64_t launches32(const Plan32& w, int64_t n);
cudaError_t launch32(const Plan32& w, const Consts32& c, const State32& A, const State32& B, const float* phi, int plane,
                     int steps, cudaStream_t stream);

// Fields of a state, as lbm_moments (outputs nr nz floats in device memory or NULL).
cudaError_t launch_fields32(const Consts32& c, const State32& A, const float* phi, int plane, float* rho, float* ur,
                            float* uz, float* T, cudaStream_t stream);

// ---- batches: one launch per step for every active instance
struct Inst32 {
    Consts32 c;
    State32 s[2];
    const float* phi;
    int plane;
};
// Blocks of a step over the instances act (parameters p, by instance number): (2 instance + kind,
// first pair or boundary node), kind 1 for boundary nodes.
struct StepBlocks {
    std::vector<int2> even, odd;   // instances with even and odd nz
};
bool serves32(const lbm_params& p);   // FP32 storage, no discrete heater
StepBlocks blocks32(const std::vector<lbm_params>& p, const std::vector<int>& act);
// lbm_rebase of the instances act[0 .. n - 1] (device memory; most_nodes: of the largest), state in
// buffer `which`.
cudaError_t launch_batch_rebase32(const Inst32* inst, const int* act, int n, int64_t most_nodes, int which,
                                  cudaStream_t stream);
cudaError_t launch_batch32(const Inst32* inst, const int2* blocks, int n, bool odd_nz, int parity, cudaStream_t stream);

}  // namespace lbm
