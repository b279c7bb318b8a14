// lbm_tile.cuh -- several time steps per launch on small grids, FP32 storage.
//
// A grid of a few thousand nodes spends its time on launches and on the latency of one node
// update after another, not on memory: a step of 48 x 96 nodes took 10.3 us in two dependent
// launches.  Here a block takes a tile of the grid with a halo as wide as the number of steps,
// holds its populations in shared memory (two buffers, one barrier per step) and advances the
// tile by up to T steps; what a step needs from outside is computed redundantly in the halo,
// so no block waits for another.  The valid part of the region shrinks by one node per step on
// the sides that are not the domain's own.
//
// What bounds it is the chain of one update (a warp alone takes about five cycles per
// instruction), so a thread takes a single node with the arithmetic of lbm_two.cuh: two nodes
// per thread in packed form took 2.1 us per step of a small block, since factors, reciprocals
// and shared-memory accesses come one per node either way.  Boundary nodes have threads of their
// own in warps behind the interior ones, so that their longer update runs beside the others': it
// pulls at the interior neighbour's place and rebuilds the boundary node's state from that
// (Sec. 4, ref. [47]).
#pragma once
#include "lbm_two.cuh"

namespace lbm {

constexpr int TILE_THREADS = 1024;   // most threads of a block (64 registers each)

// Region [a, b) of a tile [lo, lo + n) along one direction of m nodes: the halo of h on both
// sides, and the two nodes inward that a boundary node's neighbour pulls from.  Periodic
// directions wrap: the halo goes past the ends.  [ia, ib): its part without boundary nodes,
// which sit at 0 and m - 1 where the direction has them.
struct TileSpan {
    int a, b, ia, ib;
};
__host__ __device__ __forceinline__ TileSpan tile_span(int lo, int n, int h, int m, bool periodic, bool wall0) {
    const int hi = min(lo + n, m);
    TileSpan s;
    s.a = periodic ? lo - h : max(min(lo, m - 3) - h, 0);
    s.b = periodic ? hi + h : min(max(hi, 3) + h, m);
    s.ia = s.a + (!periodic && wall0 && s.a == 0 ? 1 : 0);
    s.ib = s.b - (!periodic && s.b == m ? 1 : 0);
    return s;
}
// Threads: the interior nodes, then from the next warp on the boundary nodes.
__host__ __device__ __forceinline__ int tile_inner_threads(const TileSpan& r, const TileSpan& z) {
    return ((r.ib - r.ia) * (z.ib - z.ia) + 31) & ~31;
}
__host__ __device__ __forceinline__ int tile_wall_nodes(const TileSpan& r, const TileSpan& z) {
    return (r.b - r.a) * (z.b - z.a) - (r.ib - r.ia) * (z.ib - z.ia);
}

// Boundary rebuild of one node (wall_rebuild): fh, gh, rho, ur, uz, dT hold the interior
// neighbour's pulled state (row p, reference reff, 1/phi iphf) and receive the boundary node's.
__device__ __forceinline__ void wall_node_rebuild(const Consts32& c, int p, int j, int cls, float (&fh)[9],
                                                  float (&gh)[5], float m0, float& rho, float& ur, float& uz, float& dT,
                                                  float iphf, float reff, float iphj, float refj) {
    const float rf = c.r0 + float(p), rb = c.r0 + float(j);
    const float drho = m0 * rcp_newton(rf);
    float drhob = drho, rhob = rho, urb = 0.f, uzb = 0.f;
    const bool pipe = c.geometry == PIPE_INFLOW;
    if (pipe) {   // inlet: u = (0, u_in); outlet: u of the neighbour, density 1
        const bool out = cls == OUTLET;
        urb = out ? ur : 0.f;
        uzb = out ? uz : (cls == INLET ? c.u_in : 0.f);
        drhob = out ? 0.f : drho;
        rhob = out ? 1.f : rho;
    }
    const float u2f = 1.5f * (ur * ur + uz * uz) * iphf, u2b = 1.5f * (urb * urb + uzb * uzb) * iphj;
    float mb = 0.f;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const float eu = float(ex9(i)) * ur + float(ez9(i)) * uz;
        const float q = drho + rho * (eu * (3.0f + 4.5f * iphf * eu) - u2f);
        float qb = drhob;
        if (pipe) {
            const float eb = float(ex9(i)) * urb + float(ez9(i)) * uzb;
            qb = drhob + rhob * (eb * (3.0f + 4.5f * iphj * eb) - u2b);
        }
        fh[i] = rb * w9<float>(i) * qb + fh[i] - rf * w9<float>(i) * q;
        mb += fh[i];
    }
    const float Tf = c.T0 + reff + dT;
    const float dTb = (cls == WALL_IN || cls == INLET) ? (c.T_hot - c.T0) - refj
                      : cls == WALL_OUT                ? (c.T_cold - c.T0) - refj
                                                       : (dT + reff) - refj;
    const float Tb = c.T0 + refj + dTb;
    const float tr = 0.5f * (Tb * urb - Tf * ur), tz = 0.5f * (Tb * uzb - Tf * uz);
    const float d = dTb - dT, d1 = 0.1f * d;
    gh[0] += d - 4.0f * d1;
    gh[1] += d1 + tr;
    gh[2] += d1 + tz;
    gh[3] += d1 - tr;
    gh[4] += d1 - tz;
    rho = 1.0f + mb * rcp_newton(rb);
    ur = urb;
    uz = uzb;
    dT = dTb;
}

// Advance the tile of this block by `steps` <= w.T steps from A to B.
__device__ __forceinline__ void tile_steps(const Consts32& c, const State32& A, const State32& B,
                                           const float* __restrict__ phi, int plane, const TilePlan& w, int steps,
                                           float* __restrict__ sm) {
    const int nr = c.nr, nz = c.nz;
    const bool pz = c.periodic != 0;
    const int tr = blockIdx.x / w.tiles_z, tz = blockIdx.x - tr * w.tiles_z;
    const int kr0 = tr * w.cr, kz0 = tz * w.cz;
    const bool row0_wall = c.geometry == ANNULUS || c.geometry == ANNULUS_PERIODIC_Z;
    const TileSpan sr = tile_span(kr0, w.cr, w.T, nr, false, row0_wall), sz = tile_span(kz0, w.cz, w.T, nz, pz, true);
    const int ra = sr.a, rb = sr.b, za = sz.a, zb = sz.b;   // the region (periodic z: columns modulo nz)
    const int RR = rb - ra, RZ = zb - za, RN = RR * RZ;
    float* const sR = sm;             // reference R(x)
    float* const sP = sm + RN;        // porosity
    float* const s0 = sm + 2 * RN;    // populations, two buffers of 14 planes
    const auto wrap = [&](int z) { return pz ? (z % nz + nz) % nz : z; };
    // everything above may run while the launch before this one still does
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int n = threadIdx.x; n < RN; n += blockDim.x) {
        const int y = n / RZ, x = n - y * RZ, g = (ra + y) * nz + wrap(za + x);
        sR[n] = __half2float(c.tref[g]);
        sP[n] = phi[g];
#pragma unroll
        for (int i = 0; i < 9; ++i) s0[i * RN + n] = A.f[i * plane + g];
#pragma unroll
        for (int i = 0; i < 5; ++i) s0[(9 + i) * RN + n] = A.g[i * plane + g];
    }
    __syncthreads();
    // this thread's node (j, z)
    const int t = threadIdx.x, inner = tile_inner_threads(sr, sz);
    const bool wall = t >= inner;
    bool act;
    int j, z;
    if (!wall) {
        const int IZ = sz.ib - sz.ia, y = t / IZ;
        act = y < sr.ib - sr.ia;
        j = min(sr.ia + y, sr.ib - 1);
        z = sz.ia + t - y * IZ;
    } else {   // row 0, row nr - 1, then the end columns' other rows
        int n = t - inner;
        act = n < tile_wall_nodes(sr, sz);
        const int top = (sr.ia - sr.a) * RZ, bot = (sr.b - sr.ib) * RZ, rows = sr.ib - sr.ia;
        if (n < top + bot) {
            j = n < top ? 0 : nr - 1;
            z = za + (n < top ? n : n - top);
        } else {
            n -= top + bot;
            j = sr.ia + (n < rows ? n : min(n - rows, rows - 1));
            z = sz.ia > sz.a && n < rows ? 0 : nz - 1;
        }
    }
    const int cls = wall && act ? node_class(c.geometry, nr, nz, j, wrap(z)) : FLUID;
    // the place pulled: a boundary node's interior neighbour; its sources' offsets in the region
    // (clamped into it: where that matters the node is outside the valid part)
    const int p = j == nr - 1 ? nr - 2 : (j == 0 && row0_wall ? 1 : j);
    const int q = pz ? z : min(max(z, 1), nz - 2);
    const int yp = p - ra;
    const bool axis = p == 0;   // pipe axis: the e_r = +1 sources are row 0's mirror image
    const int rm = (axis ? yp : max(yp - 1, 0)) * RZ, ro = yp * RZ, rn = min(yp + 1, RR - 1) * RZ;
    const int i1 = axis ? 3 : 1, i5 = axis ? 6 : 5, i8 = axis ? 7 : 8;
    const auto cl = [&](int x) { return min(max(x - za, 0), RZ - 1); };
    const int xo = cl(q), xm = cl(q - 1), xn = cl(q + 1), own = (j - ra) * RZ + z - za;
    // what does not change over the steps
    const float R = sR[ro + xo], ph = sP[ro + xo];
    const float t1 = 0.1f * (sR[rm + xo] - R), t3 = 0.1f * (sR[rn + xo] - R);
    const float t2 = 0.1f * (sR[ro + xm] - R), t4 = 0.1f * (sR[ro + xn] - R);
    float lin, nl, iph;
    porous_two(c, ph, lin, nl, iph);
    // the valid part loses a node per step on the sides inside the domain
    const int in_r = min(ra > 0 ? j - ra : steps, rb < nr ? rb - 1 - j : steps);
    const int in_z = min(pz || za > 0 ? z - za : steps, pz || zb < nz ? zb - 1 - z : steps);
    const int last = act ? min(in_r, in_z) : 0;   // the node is valid up to this step
    for (int s = 1; s <= steps; ++s) {
        const float* const src = s0 + ((s - 1) & 1) * 14 * RN;
        float* const dst = s0 + (s & 1) * 14 * RN;
        if (s <= last) {
            const auto ld = [&](int i, int o) { return src[i * RN + o]; };
            float fh[9], gh[5];
            fh[0] = ld(0, ro + xo);
            fh[1] = ld(i1, rm + xo);
            fh[2] = ld(2, ro + xm);
            fh[3] = ld(3, rn + xo);
            fh[4] = ld(4, ro + xn);
            fh[5] = ld(i5, rm + xm);
            fh[6] = ld(6, rn + xm);
            fh[7] = ld(7, rn + xn);
            fh[8] = ld(i8, rm + xn);
            gh[0] = ld(9, ro + xo);
            gh[1] = ld(9 + i1, rm + xo) + t1;
            gh[2] = ld(11, ro + xm) + t2;
            gh[3] = ld(12, rn + xo) + t3;
            gh[4] = ld(13, ro + xn) + t4;
            float rho, ur, uz, dT;
            Sums<float> sums = sums2(fh);
            recover_two(c, row_consts32(c, p), ph, lin, nl, sums, gh, R, rho, ur, uz, dT);
            float phj = ph, linj = lin, nlj = nl, iphj = iph, Rj = R;
            if (wall) {
                phj = sP[own];
                Rj = sR[own];
                porous_two(c, phj, linj, nlj, iphj);
                wall_node_rebuild(c, p, j, cls, fh, gh, sums.m0, rho, ur, uz, dT, iph, R, iphj, Rj);
                sums = sums2(fh);
            }
            collide_two(c, row_consts32(c, j), phj, linj, nlj, iphj, sums, fh, gh, Rj, rho, ur, uz, dT);
            if (s < steps) {
#pragma unroll
                for (int i = 0; i < 14; ++i) dst[i * RN + own] = i < 9 ? fh[i] : gh[i - 9];
            } else if (j >= kr0 && j < kr0 + w.cr && z >= kz0 && z < min(kz0 + w.cz, nz)) {
                const int g = j * nz + z;
#pragma unroll
                for (int i = 0; i < 14; ++i) (i < 9 ? B.f + i * plane : B.g + (i - 9) * plane)[g] = i < 9 ? fh[i] : gh[i - 9];
            }
        }
        if (s < steps) __syncthreads();
    }
}

}  // namespace lbm
