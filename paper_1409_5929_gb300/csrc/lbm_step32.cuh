// lbm_step32.cuh -- one time step per launch, boundary nodes included, FP32 storage.
//
// For problems whose state stays in L2 (some 10^5 to 10^6 nodes, single or as a batch) memory is
// not what bounds a step but its instructions: 563 per node in the scalar kernel of lbm.cu, about
// 250 here (two z-adjacent nodes per thread, the arithmetic of lbm_two.cuh).  A pass of two steps
// would recompute halo rows and columns, which on narrow grids costs more than the second read
// of the state saves.  Threads are numbered through the interior pairs of all rows, so no lane
// idles on a ragged row; boundary nodes take blocks of their own, one node per thread, in the
// same launch.
#pragma once
#include "lbm_tile.cuh"

namespace lbm {

constexpr int STEP_THREADS = 128;

// Rows that hold interior nodes and pairs of columns per row.
__host__ __device__ __forceinline__ int step_row0(int geometry) {
    return geometry == ANNULUS || geometry == ANNULUS_PERIODIC_Z ? 1 : 0;
}
__host__ __device__ __forceinline__ int step_pairs(int geometry, int nr, int nz) {
    return (nr - 1 - step_row0(geometry)) * ((nz + 1) / 2);
}
__host__ __device__ __forceinline__ int step_walls(int geometry, int nr, int nz) {
    return geometry == ANNULUS ? 2 * nz + 2 * (nr - 2) : geometry == ANNULUS_PERIODIC_Z ? 2 * nz
           : geometry == PIPE_INFLOW ? 2 * nr + nz - 2 : nz;
}

// Interior pair n of the problem.
template <bool VEC>
__device__ __forceinline__ void step_pair(const Consts32& c, const State32& A, const State32& B,
                                          const float* __restrict__ phi, int plane, int n) {
    const int nz = c.nz, P = (nz + 1) >> 1, y = n / P, kr = step_row0(c.geometry) + y, kz = 2 * (n - y * P);
    if (kr >= c.nr - 1) return;
    const bool pz = c.periodic != 0;
    // a lane past the last column, or on an end column of a closed problem (a boundary node),
    // computes on clamped columns and is not stored
    const bool st0 = pz || (kz > 0 && kz < nz - 1), st1 = kz + 1 < nz && (pz || kz + 1 < nz - 1);
    if (!st0 && !st1) return;
    const int lb = min(kz + 1, nz - 1);
    const int zm = kz > 0 ? kz - 1 : (pz ? nz - 1 : 0);                           // e_z = +1 source, first node
    const int zp = kz + 2 < nz ? kz + 2 : (pz ? kz + 2 - nz : nz - 1);            // e_z = -1 source, second node
    const int zp0 = kz + 1 < nz ? kz + 1 : (pz ? 0 : nz - 1);                     // and first node
    const int row = kr * nz, rowp = row + nz, rowm = kr == 0 ? row : row - nz;    // (pipe axis: mirror image)
    const int i1 = kr == 0 ? 3 : 1, i5 = kr == 0 ? 6 : 5, i8 = kr == 0 ? 7 : 8;
    const float* __restrict__ F = A.f;
    const float* __restrict__ G = A.g;
    const auto own = [&](const float* p) { return ld_two<VEC>(p, kz, lb); };
    const auto left = [&](const float* p) { return v2(__ldg(p + zm), __ldg(p + kz)); };
    const auto right = [&](const float* p) { return v2(__ldg(p + zp0), __ldg(p + zp)); };
    V2 fh[9], gh[5];
    fh[0] = own(F + row);
    fh[1] = own(F + (i1 * plane + rowm));
    fh[2] = left(F + (2 * plane + row));
    fh[3] = own(F + (3 * plane + rowp));
    fh[4] = right(F + (4 * plane + row));
    fh[5] = left(F + (i5 * plane + rowm));
    fh[6] = left(F + (6 * plane + rowp));
    fh[7] = right(F + (7 * plane + rowp));
    fh[8] = right(F + (i8 * plane + rowm));
    gh[0] = own(G + row);
    gh[1] = own(G + (i1 * plane + rowm));
    gh[2] = left(G + (2 * plane + row));
    gh[3] = own(G + (3 * plane + rowp));
    gh[4] = right(G + (4 * plane + row));
    const V2 ph = own(phi + row);
    const auto ref = [&](int o, int a, int b) {
        return v2(__half2float(__ldg(c.tref + o + a)), __half2float(__ldg(c.tref + o + b)));
    };
    const V2 R = ref_of(ld_ref<VEC>(c.tref + row, kz, lb));
    gh[1] += (ref_of(ld_ref<VEC>(c.tref + rowm, kz, lb)) - R) * both(0.1f);
    gh[2] += (ref(row, zm, kz) - R) * both(0.1f);
    gh[3] += (ref_of(ld_ref<VEC>(c.tref + rowp, kz, lb)) - R) * both(0.1f);
    gh[4] += (ref(row, zp0, zp) - R) * both(0.1f);
    const Row32 q = row_consts32(c, kr);
    V2 lin, nl, iph, rho, ur, uz, dT;
    porous_two(c, ph, lin, nl, iph);
    const Sums<V2> sums = sums2(fh);
    recover_two(c, q, ph, lin, nl, sums, gh, R, rho, ur, uz, dT);
    collide_two(c, q, ph, lin, nl, iph, sums, fh, gh, R, rho, ur, uz, dT);
    float* __restrict__ Fo = B.f + row + kz;
    float* __restrict__ Go = B.g + row + kz;
    if (st0 && st1) {
#pragma unroll
        for (int i = 0; i < 9; ++i) st_two<VEC>(Fo + i * plane, fh[i], true);
#pragma unroll
        for (int i = 0; i < 5; ++i) st_two<VEC>(Go + i * plane, gh[i], true);
    } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) Fo[i * plane + (st0 ? 0 : 1)] = st0 ? fh[i].v.x : fh[i].v.y;
#pragma unroll
        for (int i = 0; i < 5; ++i) Go[i * plane + (st0 ? 0 : 1)] = st0 ? gh[i].v.x : gh[i].v.y;
    }
}

// Boundary node n of the problem: the numbering of wall_node (lbm.cu).
__device__ __forceinline__ void step_wall(const Consts32& c, const State32& A, const State32& B,
                                          const float* __restrict__ phi, int plane, int n) {
    const int nr = c.nr, nz = c.nz;
    const bool pz = c.periodic != 0, row0_wall = step_row0(c.geometry) != 0;
    int j, z;
    if (c.geometry == PIPE_INFLOW) {   // inlet, outlet, wall without the corners
        j = n < 2 * nr ? (n < nr ? n : n - nr) : nr - 1;
        z = n < 2 * nr ? (n < nr ? 0 : nz - 1) : 1 + n - 2 * nr;
    } else {                           // wall rows, then bottom and top without the corners
        const int rows = (row0_wall ? 2 : 1) * nz;
        if (n < rows) {
            j = row0_wall && n < nz ? 0 : nr - 1;
            z = row0_wall && n >= nz ? n - nz : n;
        } else {
            const int m = n - rows;
            j = 1 + (m < nr - 2 ? m : m - (nr - 2));
            z = m < nr - 2 ? 0 : nz - 1;
        }
    }
    const int cls = node_class(c.geometry, nr, nz, j, z);
    // the place pulled: the interior neighbour
    const int p = j == nr - 1 ? nr - 2 : (j == 0 && row0_wall ? 1 : j), q = pz ? z : min(max(z, 1), nz - 2);
    const int qm = q > 0 ? q - 1 : nz - 1, qp = q < nz - 1 ? q + 1 : 0;
    const int row = p * nz, rowp = row + nz, rowm = p == 0 ? row : row - nz, own = j * nz + z;
    const int i1 = p == 0 ? 3 : 1, i5 = p == 0 ? 6 : 5, i8 = p == 0 ? 7 : 8;
    const auto f = [&](int i, int o) { return __ldg(A.f + i * plane + o); };
    const auto g = [&](int i, int o) { return __ldg(A.g + i * plane + o); };
    const auto ref = [&](int o) { return __half2float(__ldg(c.tref + o)); };
    float fh[9] = {f(0, row + q), f(i1, rowm + q), f(2, row + qm), f(3, rowp + q), f(4, row + qp),
                   f(i5, rowm + qm), f(6, rowp + qm), f(7, rowp + qp), f(i8, rowm + qp)};
    const float R = ref(row + q), Rj = ref(own), ph = __ldg(phi + row + q), phj = __ldg(phi + own);
    float gh[5] = {g(0, row + q), g(i1, rowm + q) + 0.1f * (ref(rowm + q) - R), g(2, row + qm) + 0.1f * (ref(row + qm) - R),
                   g(3, rowp + q) + 0.1f * (ref(rowp + q) - R), g(4, row + qp) + 0.1f * (ref(row + qp) - R)};
    float lin, nl, iph, rho, ur, uz, dT;
    porous_two(c, ph, lin, nl, iph);
    Sums<float> sums = sums2(fh);
    recover_two(c, row_consts32(c, p), ph, lin, nl, sums, gh, R, rho, ur, uz, dT);
    float linj, nlj, iphj;
    porous_two(c, phj, linj, nlj, iphj);
    wall_node_rebuild(c, p, j, cls, fh, gh, sums.m0, rho, ur, uz, dT, iph, R, iphj, Rj);
    sums = sums2(fh);
    collide_two(c, row_consts32(c, j), phj, linj, nlj, iphj, sums, fh, gh, Rj, rho, ur, uz, dT);
#pragma unroll
    for (int i = 0; i < 9; ++i) B.f[i * plane + own] = fh[i];
#pragma unroll
    for (int i = 0; i < 5; ++i) B.g[i * plane + own] = gh[i];
}

}  // namespace lbm
