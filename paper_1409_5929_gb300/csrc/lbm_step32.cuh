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

// Interior pair n of the problem, pulled: the first of its two nodes, which of them are interior
// nodes, their pre-collision deviations, porosity and temperature reference.  False: neither is.
struct PairNode {
    int kr, kz;
    bool st0, st1;
    V2 f[9], g[5], ph, R;
};
template <bool VEC>
__device__ __forceinline__ bool pull_pair(const Consts32& c, const State32& A, const float* __restrict__ phi, int plane,
                                          int n, PairNode& v) {
    const int nz = c.nz, P = (nz + 1) >> 1, y = n / P, kr = step_row0(c.geometry) + y, kz = 2 * (n - y * P);
    if (kr >= c.nr - 1) return false;
    const bool pz = c.periodic != 0;
    // a lane past the last column, or on an end column of a closed problem (a boundary node),
    // computes on clamped columns and is not stored
    v.kr = kr;
    v.kz = kz;
    v.st0 = pz || (kz > 0 && kz < nz - 1);
    v.st1 = kz + 1 < nz && (pz || kz + 1 < nz - 1);
    if (!v.st0 && !v.st1) return false;
    const int lb = min(kz + 1, nz - 1);
    const int zm = kz > 0 ? kz - 1 : (pz ? nz - 1 : 0);                           // e_z = +1 source, first node
    const int zp = kz + 2 < nz ? kz + 2 : (pz ? kz + 2 - nz : nz - 1);            // e_z = -1 source, second node
    const int zp0 = kz + 1 < nz ? kz + 1 : (pz ? 0 : nz - 1);                     // and first node
    const int row = kr * nz, rowp = row + nz, rowm = kr == 0 ? row : row - nz;    // (pipe axis: mirror image)
    const int i1 = kr == 0 ? 3 : 1, i5 = kr == 0 ? 6 : 5, i8 = kr == 0 ? 7 : 8;
    const float* __restrict__ F = A.f;
    const float* __restrict__ G = A.g;
    const auto own = [&](const float* p) { return ld_two<VEC>(p, kz, lb); };
    const auto left = [&](const float* p) { return v2(p[zm], p[kz]); };
    const auto right = [&](const float* p) { return v2(p[zp0], p[zp]); };
    v.f[0] = own(F + row);
    v.f[1] = own(F + (i1 * plane + rowm));
    v.f[2] = left(F + (2 * plane + row));
    v.f[3] = own(F + (3 * plane + rowp));
    v.f[4] = right(F + (4 * plane + row));
    v.f[5] = left(F + (i5 * plane + rowm));
    v.f[6] = left(F + (6 * plane + rowp));
    v.f[7] = right(F + (7 * plane + rowp));
    v.f[8] = right(F + (i8 * plane + rowm));
    v.g[0] = own(G + row);
    v.g[1] = own(G + (i1 * plane + rowm));
    v.g[2] = left(G + (2 * plane + row));
    v.g[3] = own(G + (3 * plane + rowp));
    v.g[4] = right(G + (4 * plane + row));
    v.ph = own(phi + row);
    const auto ref = [&](int o, int a, int b) {
        return v2(__half2float(c.tref[o + a]), __half2float(c.tref[o + b]));
    };
    v.R = ref_of(ld_ref<VEC>(c.tref + row, kz, lb));
    v.g[1] += (ref_of(ld_ref<VEC>(c.tref + rowm, kz, lb)) - v.R) * both(0.1f);
    v.g[2] += (ref(row, zm, kz) - v.R) * both(0.1f);
    v.g[3] += (ref_of(ld_ref<VEC>(c.tref + rowp, kz, lb)) - v.R) * both(0.1f);
    v.g[4] += (ref(row, zp0, zp) - v.R) * both(0.1f);
    return true;
}

template <bool VEC>
__device__ __forceinline__ void step_pair(const Consts32& c, const State32& A, const State32& B,
                                          const float* __restrict__ phi, int plane, int n) {
    PairNode v;
    if (!pull_pair<VEC>(c, A, phi, plane, n, v)) return;
    const Row32 q = row_consts32(c, v.kr);
    V2 lin, nl, iph, rho, ur, uz, dT;
    porous_two(c, v.ph, lin, nl, iph);
    const Sums<V2> sums = sums2(v.f);
    recover_two(c, q, v.ph, lin, nl, sums, v.g, v.R, rho, ur, uz, dT);
    collide_two(c, q, v.ph, lin, nl, iph, sums, v.f, v.g, v.R, rho, ur, uz, dT);
    float* __restrict__ Fo = B.f + v.kr * c.nz + v.kz;
    float* __restrict__ Go = B.g + v.kr * c.nz + v.kz;
    if (v.st0 && v.st1) {
#pragma unroll
        for (int i = 0; i < 9; ++i) st_two<VEC>(Fo + i * plane, v.f[i], true);
#pragma unroll
        for (int i = 0; i < 5; ++i) st_two<VEC>(Go + i * plane, v.g[i], true);
    } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) Fo[i * plane + (v.st0 ? 0 : 1)] = v.st0 ? v.f[i].v.x : v.f[i].v.y;
#pragma unroll
        for (int i = 0; i < 5; ++i) Go[i * plane + (v.st0 ? 0 : 1)] = v.st0 ? v.g[i].v.x : v.g[i].v.y;
    }
}

// Where fields go: rho, u_r, u_z, T, each nr nz or NULL; vec: pairs of them may be stored as one
// (8-byte aligned, even nz).
struct Fields {
    float* p[4];
    int vec;
};
Fields fields_of(int nz, float* rho, float* ur, float* uz, float* T);   // (lbm_f32.cu)
__device__ __forceinline__ void put_pair(const Fields& o, int at, bool st0, bool st1, V2 rho, V2 ur, V2 uz, V2 T) {
    const V2 v[4] = {rho, ur, uz, T};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (!o.p[k]) continue;
        if (o.vec && st0 && st1) {
            *reinterpret_cast<float2*>(o.p[k] + at) = v[k].v;
        } else {
            if (st0) o.p[k][at] = v[k].v.x;
            if (st1) o.p[k][at + 1] = v[k].v.y;
        }
    }
}
template <bool VEC>
__device__ __forceinline__ void fields_pair(const Consts32& c, const State32& A, const float* __restrict__ phi, int plane,
                                            int n, const Fields& o) {
    PairNode v;
    if (!pull_pair<VEC>(c, A, phi, plane, n, v)) return;
    V2 lin, nl, iph, rho, ur, uz, dT;
    porous_two(c, v.ph, lin, nl, iph);
    recover_two(c, row_consts32(c, v.kr), v.ph, lin, nl, sums2(v.f), v.g, v.R, rho, ur, uz, dT);
    put_pair(o, v.kr * c.nz + v.kz, v.st0, v.st1, rho, ur, uz, (v.R + both(c.T0)) + dT);
}

// Boundary node n of the problem: the numbering of wall_node (lbm.cu).
// STEP: its update stored in B; else its fields.
template <bool STEP>
__device__ __forceinline__ void step_wall(const Consts32& c, const State32& A, const State32& B,
                                          const float* __restrict__ phi, int plane, int n, const Fields& o) {
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
    const auto f = [&](int i, int o) { return A.f[i * plane + o]; };
    const auto g = [&](int i, int o) { return A.g[i * plane + o]; };
    const auto ref = [&](int o) { return __half2float(c.tref[o]); };
    float fh[9] = {f(0, row + q), f(i1, rowm + q), f(2, row + qm), f(3, rowp + q), f(4, row + qp),
                   f(i5, rowm + qm), f(6, rowp + qm), f(7, rowp + qp), f(i8, rowm + qp)};
    const float R = ref(row + q), Rj = ref(own), ph = phi[row + q], phj = phi[own];
    float gh[5] = {g(0, row + q), g(i1, rowm + q) + 0.1f * (ref(rowm + q) - R), g(2, row + qm) + 0.1f * (ref(row + qm) - R),
                   g(3, rowp + q) + 0.1f * (ref(rowp + q) - R), g(4, row + qp) + 0.1f * (ref(row + qp) - R)};
    float lin, nl, iph, rho, ur, uz, dT;
    porous_two(c, ph, lin, nl, iph);
    Sums<float> sums = sums2(fh);
    recover_two(c, row_consts32(c, p), ph, lin, nl, sums, gh, R, rho, ur, uz, dT);
    float linj, nlj, iphj;
    porous_two(c, phj, linj, nlj, iphj);
    wall_node_rebuild(c, p, j, cls, fh, gh, sums.m0, rho, ur, uz, dT, iph, R, iphj, Rj);
    if (!STEP) {
        const float v[4] = {rho, ur, uz, (c.T0 + Rj) + dT};
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (o.p[k]) o.p[k][own] = v[k];
        return;
    }
    sums = sums2(fh);
    collide_two(c, row_consts32(c, j), phj, linj, nlj, iphj, sums, fh, gh, Rj, rho, ur, uz, dT);
#pragma unroll
    for (int i = 0; i < 9; ++i) B.f[i * plane + own] = fh[i];
#pragma unroll
    for (int i = 0; i < 5; ++i) B.g[i * plane + own] = gh[i];
}

}  // namespace lbm
