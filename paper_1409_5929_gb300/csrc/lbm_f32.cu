// lbm_f32.cu -- kernels and host side of lbm_f32.h: several time steps per launch, FP32 storage.
#include "lbm_f32.h"

#include <algorithm>
#include <cmath>

#include "lbm_dependent.h"
#include "lbm_step32.cuh"
#include "lbm_tile.cuh"
#include "lbm_two.cuh"

using namespace lbm;

// Two steps per pass (lbm_two.cuh): one warp per strip of columns and chunk of rows; warps are
// independent.  At 4096 x 8192 a pass takes 0.68 ms for two steps where two single steps take
// 1.24 ms (0.60 ms each, 97 % of the copy bandwidth, and the wall kernel): it moves the state's
// 118 bytes per node once, at 86 % of the copy bandwidth, and issues 260 instructions per node
// and step (563 in k_bulk).  128 registers, four blocks per SM; with five many more of them spill,
// with three too few warps are in flight.  Per step of a long run with three / four / five blocks:
// 4096 x 8192 0.366 / 0.344 / 0.478 ms; odd nz, 4095 x 8191 (two loads per pair, 92 bytes spilled at
// four blocks against 16) 0.398 / 0.379 / 0.590 ms, single steps of k_bulk 0.688.  The marches that
// meet boundary nodes (the end strips, the first and the last chunk of every strip, the wall rows) come
// first and run a form of the march of their own: the boundary rebuild between a row's recovery and its
// collision cost the other marches 13 % (4096 x 8192, FP32) when one form served both.
#ifndef LBM_TWO_MIN_BLOCKS
#define LBM_TWO_MIN_BLOCKS 4
#endif
template <bool VEC>
__global__ void __launch_bounds__(TWO_THREADS, LBM_TWO_MIN_BLOCKS) k_two(const Consts32 c, const State32 A,
                                                                         const State32 B,
                                                                         const float* phi, int plane,
                                                                         const TwoPlan w) {
    __shared__ float4 ring[TWO_KEEP * TWO_THREADS];
    constexpr int WARPS = TWO_THREADS / 32;
    const int wall_blocks = (w.n_wall() + WARPS - 1) / WARPS, warp = threadIdx.x >> 5;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if ((int)blockIdx.x >= wall_blocks) {
        const int t = ((int)blockIdx.x - wall_blocks) * WARPS + warp;
        if (t >= w.n_bulk()) return;
        const int chunk = t / w.inner(), lo = w.first + w.erows + chunk * w.rows;
        two_march<VEC, false>(c, A, B, phi, plane, 1 + t - chunk * w.inner(), lo,
                                   min(lo + w.rows - 1, w.last - w.erows), -1, ring);
        return;
    }
    int t = blockIdx.x * WARPS + warp, s, lo, hi, wall = -1;
    if (t < w.ends() * w.echunks()) {
        const int chunk = t / w.ends();
        s = t - chunk * w.ends() == 0 ? 0 : w.strips - 1;
        lo = w.first + chunk * w.erows;
        hi = min(lo + w.erows - 1, w.last);
    } else if ((t -= w.ends() * w.echunks()) < w.inner() * w.outer()) {
        const int chunk = t / w.inner();
        s = 1 + t - chunk * w.inner();
        lo = chunk == 0 ? w.first : max(w.last - w.erows + 1, w.first + w.erows);
        hi = chunk == 0 ? min(w.first + w.erows - 1, w.last) : w.last;
    } else {
        t -= w.inner() * w.outer();
        const int k = t / w.strips;
        if (k >= w.walls()) return;
        s = t - k * w.strips;
        wall = k == 0 ? c.nr - 1 : 0;
        lo = hi = wall ? w.last : 1;
    }
    two_march<VEC, true>(c, A, B, phi, plane, s, lo, hi, wall, ring);
}

// One step of every node (lbm_step32.cuh): the blocks of the boundary nodes first, so that their
// longer chain starts early.  512 x 1024: 8.1 us per step (19.0 with k_bulk and k_wall, 563
// instructions per node against about 250); 4096 x 8192: 0.60 ms, as k_bulk, without k_wall's 14 us.
// 80 registers, six blocks per SM; with eight (64 registers) they spill, 9.4 us.
#ifndef LBM_STEP_MIN_BLOCKS
#define LBM_STEP_MIN_BLOCKS 6
#endif
template <bool VEC>
__global__ void __launch_bounds__(STEP_THREADS, LBM_STEP_MIN_BLOCKS) k_step(const Consts32 c, const State32 A,
                                                                            const State32 B,
                                                                            const float* phi, int plane,
                                                                            int walls) {
    const int wall_blocks = (walls + STEP_THREADS - 1) / STEP_THREADS;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if ((int)blockIdx.x < wall_blocks) {
        const int n = blockIdx.x * STEP_THREADS + threadIdx.x;
        if (n < walls) step_wall<true>(c, A, B, phi, plane, n, Fields{});
    } else {
        step_pair<VEC>(c, A, B, phi, plane, ((int)blockIdx.x - wall_blocks) * STEP_THREADS + threadIdx.x);
    }
}
// The fields of a state (what the next step's pull sees).  Against k_moments (one node per thread and
// the boundary rebuild in the same warps): one step of 48 x 96 and its fields 8.2 -> 7.1 us,
// 4096 x 8192 0.42 -> 0.36 ms (FP16 storage, k_fields16: 0.48 -> 0.36).  Blocks per SM 8 / 9 / 10 / 11:
// 4096 x 8192 372 / 368 / 364 / 376 us, 512 x 1024 5.63 / 5.54 / 5.48 / 6.47; odd nz, 4095 x 8191
// 394 / 389 / 398 / 432, 1023 x 2047 27.2 / 26.9 / 28.5 / 31.7.
template <bool VEC>
__global__ void __launch_bounds__(STEP_THREADS, VEC ? 10 : 9) k_fields(const Consts32 c, const State32 A, const float* phi,
                                                            int plane, int walls, const Fields o) {
    const int wall_blocks = (walls + STEP_THREADS - 1) / STEP_THREADS;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if ((int)blockIdx.x < wall_blocks) {
        const int n = blockIdx.x * STEP_THREADS + threadIdx.x;
        if (n < walls) step_wall<false>(c, A, A, phi, plane, n, o);
    } else {
        fields_pair<VEC>(c, A, phi, plane, ((int)blockIdx.x - wall_blocks) * STEP_THREADS + threadIdx.x, o);
    }
}
// The same for a batch: a block's instance (kind 1: boundary nodes) and its first pair or node; the
// instance's constants are read from shared memory.  16 instances of 64 to 160 rows (450 k nodes):
// 8.5 us per step (14 as a graph of k_batch_bulk and the forked k_batch_wall; 12.5 with two-step
// marches, whose halos cost more than they save on rows of 128 to 320 columns).
template <bool VEC>
__global__ void __launch_bounds__(STEP_THREADS, LBM_STEP_MIN_BLOCKS) k_batch_step(const Inst32* __restrict__ inst,
                                                                                  const int2* __restrict__ blocks,
                                                                                  int parity) {
    __shared__ Inst32 d;
    const int2 b = blocks[blockIdx.x];   // the lists and constants are not written by a launch
    for (int w = threadIdx.x; w < (int)(sizeof(Inst32) / sizeof(int)); w += STEP_THREADS)
        reinterpret_cast<int*>(&d)[w] = reinterpret_cast<const int*>(inst + (b.x >> 1))[w];
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int n = b.y + threadIdx.x;
    if (b.x & 1) {
        if (n < step_walls(d.c.geometry, d.c.nr, d.c.nz)) step_wall<true>(d.c, d.s[parity], d.s[parity ^ 1], d.phi, d.plane, n, Fields{});
    } else {
        step_pair<VEC>(d.c, d.s[parity], d.s[parity ^ 1], d.phi, d.plane, n);
    }
}

// Reference refresh (rebase_thermal_node of lbm.cu) of the instances act[blockIdx.y]: R(x) becomes the
// temperature offset of the state in buffer `which`, the stored temperatures are re-expressed against it.  One
// launch for the batch: 16 launches of k_rebase took 73 us.  Blocks per instance for four nodes per thread
// of the largest one, as many as k_rebase's 4096 at most (64 each left most of the device idle on one or
// two large instances: 1 x 4096 x 4096 8134 against 7573 us per check, 1 x 1500 x 3000 2192 against 2040).
__global__ void __launch_bounds__(256) k_batch_rebase(const Inst32* __restrict__ inst, const int* __restrict__ act, int which) {
    const Inst32& d = inst[act[blockIdx.y]];
    const int N = d.c.nr * d.c.nz, plane = d.plane;
    float* const G = d.s[which].g;
    __half* const ref = const_cast<__half*>(d.c.tref);
    for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < N; n += gridDim.x * blockDim.x) {
        float g[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) g[i] = G[i * plane + n];
        const float r_old = __half2float(ref[n]);
        const float t = r_old + (((g[0] + g[1]) + (g[2] + g[3])) + g[4]);
        const __half h = __float2half_rn(fminf(fmaxf(t, -60000.f), 60000.f));
        const float e = r_old - __half2float(h), e1 = 0.1f * e;
        G[n] = g[0] + (e - 4.f * e1);
#pragma unroll
        for (int i = 1; i < 5; ++i) G[i * plane + n] = g[i] + e1;
        ref[n] = h;
    }
}

// Several steps per launch on small grids (lbm_tile.cuh).  48 x 96: 1.5 us per step (10.3 as two
// launches per step, 4.7 with k_two; 1.9 without the dependent launch); 100 x 200: 1.7 us.
__global__ void __launch_bounds__(TILE_THREADS, 1) k_tile(const Consts32 c, const State32 A,
                                                          const State32 B, const float* phi,
                                                          int plane, const TilePlan w, int steps) {
    extern __shared__ float tile_sm[];
    tile_steps(c, A, B, phi, plane, w, steps, tile_sm);
}

// Rows per march of k_two.  A march of r rows takes r + 2 first and r second steps, so long
// marches waste least, short ones fill the device: the r with the least (r + 2.5) x waves of
// resident warps, half a wave added for the last one where there is more than one.  (4096 x
// 8192, FP32: r = 32, 0.340 ms per step; 64 rows 0.355, 16 rows 0.343.)  The pipe's axis row
// belongs to marches of the boundary form, so those take two rows there at least.
static TwoPlan two_plan(const lbm_params& p, int sms) {
    TwoPlan w, best = {};
    w.first = (p.geometry == LBM_ANNULUS || p.geometry == LBM_ANNULUS_PERIODIC_Z) ? 1 : 0;
    w.last = p.nr - 2;
    w.strips = ((periodic_z(p.geometry) ? p.nz : p.nz & ~1) + TWO_COLS - 1) / TWO_COLS;
    const double slots = (double)sms * LBM_TWO_MIN_BLOCKS * (TWO_THREADS / 32);
    double cost = INFINITY;
    for (int r = 1; r <= 256; ++r) {
        w.rows = r;
        w.erows = std::max(r * 5 / 8, w.first ? 1 : 2);
        const double waves = (w.n_wall() + w.n_bulk()) / slots;
        const double t = (r + 2.5) * (waves <= 1 ? 1.0 : waves + 0.5);
        if (t < cost) { cost = t; best = w; }
        if (r > w.last - w.first) break;
    }
    return best;
}

// Tile and steps per launch of k_tile: the least estimated time per step, from measured launches
// (us): 4.1 for a launch with the loads and stores of the tile (2.6 + 1.5 per wave), and a step of a
// block 1.1, the chain of one update, or 0.28 per four warps on the SM where those take longer.
// 48 x 96 gets 8 steps of 4 x 8 tiles (144 blocks), 100 x 200 5 steps of 10 x 14 (150 blocks).
static TilePlan tile_plan(const lbm_params& p, int sms) {
    TilePlan w = {}, best = {};
    double cost = INFINITY;
    const bool pz = periodic_z(p.geometry);
    const bool wall0 = p.geometry == LBM_ANNULUS || p.geometry == LBM_ANNULUS_PERIODIC_Z;
    // the largest region along a direction for each number of its boundary rows (0, 1 or 2): those
    // next to the ends and one from the middle
    struct Spans { TileSpan s[3]; };
    const auto size = [](const TileSpan& s) { return s.b - s.a; };
    const auto spans = [&](int n, int h, int m, bool periodic, bool wall0) {
        Spans out = {};
        const int tiles = (m + n - 1) / n, k = h / n + 3;
        for (int i = 0; i < tiles; i = (i == k && tiles - k > k + 1) ? tiles - k : i + 1) {
            const TileSpan s = tile_span(i * n, n, h, m, periodic, wall0);
            TileSpan& o = out.s[size(s) - (s.ib - s.ia)];
            if (size(s) > size(o)) o = s;
        }
        return out;
    };
    static const int sizes[] = {2,  3,  4,  5,  6,  7,  8,  9,  10, 11, 12, 14, 16, 18,
                                20, 22, 24, 26, 28, 30, 32, 36, 40, 48, 56, 64, 96, 128};
    constexpr int NS = sizeof(sizes) / sizeof(int);
    const double share = (double)p.nr * p.nz / sms;   // nodes per SM: tiles from a third of that on
    for (int T : {8, 10, 6, 5, 4, 3, 2}) {
        if ((4.1 + 1.1 * T) / T >= cost) continue;    // no tile can beat the best one found
        Spans vz[NS];
        int nz = 0;
        for (; nz < NS && sizes[nz] <= p.nz + 2; ++nz) vz[nz] = spans(sizes[nz], T, p.nz, pz, true);
        for (int cr : sizes) {
            if (cr > std::min(64, p.nr)) break;
            const Spans vr = spans(cr, T, p.nr, false, wall0);
            for (int i = 2; i < nz; ++i) {
                if (3 * cr * sizes[i] < share) continue;
                if (cr * sizes[i] > 1.2 * share + 8) break;
                w.T = T;
                w.cr = cr;
                w.cz = sizes[i];
                int threads = 0, nodes = 0;
                for (const auto& r : vr.s)
                    for (const auto& z : vz[i].s) {
                        if (!size(r) || !size(z)) continue;
                        threads = std::max(threads, tile_inner_threads(r, z) + tile_wall_nodes(r, z));
                        nodes = std::max(nodes, size(r) * size(z));
                    }
                w.threads = (threads + 31) / 32 * 32;
                if (w.threads > TILE_THREADS) break;
                w.shared = (size_t)30 * nodes * sizeof(float);
                w.tiles_z = (p.nz + w.cz - 1) / w.cz;
                w.blocks = ((p.nr + cr - 1) / cr) * w.tiles_z;
                const int fit = std::max(1, std::min(TILE_THREADS / w.threads, (int)(220000 / w.shared)));
                const double per_sm = std::ceil((double)w.blocks / sms);
                const double waves = std::ceil(per_sm / fit), busy = std::min<double>(per_sm, fit) * w.threads / 128.0;
                const double t_launch = 2.6 + waves * (1.5 + T * std::max(1.1, 0.28 * busy));
                if (t_launch / T < cost) { cost = t_launch / T; best = w; }
            }
        }
    }
    return best;
}

namespace lbm {

Consts32 consts32(const Consts<double>& d, const Consts<float>& f) {
    Consts32 c;
    static_cast<Consts<float>&>(c) = f;
    c.a_e = (float)(d.s_e / 36);
    c.g_u = (float)(d.s_e / 12);
    c.g_f = (float)(d.h_e / 6);
    c.a_j = (float)(d.s_j / 6);
    c.b_j = (float)(d.h_j / 6);
    c.a_q = (float)(d.s_q / 12);
    c.b_q = (float)(d.h_q / 12);
    c.a_nu = (float)(d.s_nu / 4);
    c.b7 = (float)(d.h_nu / 2);
    c.b8 = (float)(d.h_nu / 4);
    return c;
}

// k_tile up to this many nodes, k_step above: where their times per step of a long run cross (k_tile
// against k_step: 200 x 400 2.9 / 4.6 us, 250 x 500 4.2 / 5.9, 300 x 600 5.5 / 5.6, 350 x 600 6.7 / 5.6,
// 400 x 625 7.7 / 6.4).  Calls of one or two steps, which load a halo for the longest launch, would
// cross near 100 x 200 already (3.9 / 3.7 us; 200 x 400 5.7 / 4.4, 300 x 600 10.1 / 5.7); before k_tile
// such a step took two launches, 10.4 to 12.5 us.
constexpr int64_t TILE_MAX_NODES = 200000;

// One step per launch up to this many nodes, where the state stays in L2 (both buffers 112 bytes per
// node), two steps per launch above (k_step against k_two): 512 x 1024 8.1 against 11.1 us per step,
// 700 x 1400 17.3 against 18.0, 1000 x 1500 29.3 against 24.6.
constexpr int64_t STEP_MAX_NODES = 1000000;

cudaError_t plan32(const lbm_params& p, int sms, Plan32* out) {
    out->two = two_plan(p, sms);
    out->tile = TilePlan{};
    out->single = (int64_t)p.nr * p.nz <= STEP_MAX_NODES;
    if ((int64_t)p.nr * p.nz > TILE_MAX_NODES) return cudaSuccess;
    out->tile = tile_plan(p, sms);
    return cudaFuncSetAttribute(k_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}

int steps32(const Plan32& w, int64_t left) {
    if (w.tile.T) return (int)std::max<int64_t>(1, std::min<int64_t>(w.tile.T, left - 1));
    return w.two.strips && left >= 3 && !w.single ? 2 : 1;
}

int64_t launches32(const Plan32& w, int64_t n) {
    int64_t k = 0;
    for (; n > 0; ++k) n -= steps32(w, n);
    return k;
}

cudaError_t launch32(const Plan32& w, const Consts32& c, const State32& A, const State32& B, const float* phi, int plane,
                     int steps, cudaStream_t stream) {
    if (w.tile.T)
        return launch_dependent(k_tile, w.tile.blocks, w.tile.threads, w.tile.shared, stream, c, A, B, phi, plane, w.tile,
                                steps);
    if (steps == 1) {
        const int walls = step_walls(c.geometry, c.nr, c.nz), pairs = step_pairs(c.geometry, c.nr, c.nz);
        const unsigned blocks = (walls + STEP_THREADS - 1) / STEP_THREADS + (pairs + STEP_THREADS - 1) / STEP_THREADS;
        return launch_dependent(c.nz & 1 ? k_step<false> : k_step<true>, blocks, STEP_THREADS, 0, stream, c, A, B, phi,
                                plane, walls);
    }
    constexpr int WARPS = TWO_THREADS / 32;
    const unsigned blocks = (unsigned)((w.two.n_wall() + WARPS - 1) / WARPS + (w.two.n_bulk() + WARPS - 1) / WARPS);
    return launch_dependent(c.nz & 1 ? k_two<false> : k_two<true>, blocks, TWO_THREADS, 0, stream, c, A, B, phi, plane,
                            w.two);
}

bool serves32(const lbm_params& p) { return p.storage == LBM_F32 && !(p.heater_len > 0); }

StepBlocks blocks32(const std::vector<lbm_params>& p, const std::vector<int>& act) {
    StepBlocks out;
    for (int kind = 1; kind >= 0; --kind)
        for (int i : act) {
            const int n = kind ? step_walls(p[i].geometry, p[i].nr, p[i].nz) : step_pairs(p[i].geometry, p[i].nr, p[i].nz);
            for (int k = 0; k < n; k += STEP_THREADS) ((p[i].nz & 1) ? out.odd : out.even).push_back(make_int2(2 * i + kind, k));
        }
    return out;
}

cudaError_t launch_batch32(const Inst32* inst, const int2* blocks, int n, bool odd_nz, int parity, cudaStream_t stream) {
    return launch_dependent(odd_nz ? k_batch_step<false> : k_batch_step<true>, (unsigned)n, STEP_THREADS, 0, stream, inst,
                            blocks, parity);
}

Fields fields_of(int nz, float* rho, float* ur, float* uz, float* T) {
    Fields o = {{rho, ur, uz, T}, (nz & 1) == 0};
    for (const float* p : o.p) o.vec = o.vec && ((uintptr_t)p & 7) == 0;
    return o;
}

cudaError_t launch_fields32(const Consts32& c, const State32& A, const float* phi, int plane, float* rho, float* ur,
                            float* uz, float* T, cudaStream_t stream) {
    const int walls = step_walls(c.geometry, c.nr, c.nz), pairs = step_pairs(c.geometry, c.nr, c.nz);
    const unsigned blocks = (walls + STEP_THREADS - 1) / STEP_THREADS + (pairs + STEP_THREADS - 1) / STEP_THREADS;
    return launch_dependent(c.nz & 1 ? k_fields<false> : k_fields<true>, blocks, STEP_THREADS, 0, stream, c, A, phi, plane,
                            walls, fields_of(c.nz, rho, ur, uz, T));
}

cudaError_t launch_batch_rebase32(const Inst32* inst, const int* act, int n, int64_t most_nodes, int which,
                                  cudaStream_t stream) {
    const unsigned blocks = (unsigned)std::min<int64_t>((most_nodes + 1023) / 1024, 4096);
    k_batch_rebase<<<dim3(blocks, (unsigned)n), 256, 0, stream>>>(inst, act, which);
    return cudaGetLastError();
}

}  // namespace lbm
