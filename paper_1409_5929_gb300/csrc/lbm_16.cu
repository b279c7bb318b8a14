// lbm_16.cu -- kernels and host side of lbm_16.h.
#include "lbm_16.h"

#include <vector>

#include "lbm_dependent.h"
#include "lbm_nodes.cuh"
#include "lbm_step32.cuh"

using namespace lbm;

template <int STO> static __device__ __forceinline__ Buf<STO> buf16(const Step16& s, int which) {
    Buf<STO> b;
    b.f = (typename St<STO>::TF*)s.f[which];
    b.g = s.g[which];
    return b;
}

// Boundary node n (the update of k_wall).
template <int STO>
__device__ __forceinline__ void wall16(const Consts<float>& c, const Buf<STO>& A, const Buf<STO>& B,
                                       const float* __restrict__ phi, int64_t plane, int n) {
    int kr, kz;
    wall_node(c.geometry, c.nr, c.nz, n, kr, kz);
    const int cls = node_class(c.geometry, c.nr, c.nz, kr, kz);
    float fh[9], gh[5], m0, rho, urb, uzb, dTb, refb;
    wall_state<STO, float, LAY_N, true>(c, A, phi, plane, cls, kr, kz, fh, gh, m0, rho, urb, uzb, dTb, refb);
    const int64_t m = (int64_t)kr * c.nz + kz;
    const float r = c.r0 + float(kr), ph = ldv<true>(phi + m);
    float lin, nl, iph;
    porous(c, ph, lin, nl, iph);
    collide(c, r, rcp_acc(r), ph, lin, nl, iph, fh, gh, refb, m0, rho, urb, uzb, dTb);
    store<STO>(c, B, plane, kr, kz, m, fh, gh);
}

// Odd nz, closed in z: rows start at alternating alignment, so a row's pairs start at its first
// 4-byte-aligned element (column 0 or -1).  Then the pair itself and the diagonal sources (row +- 1,
// column +- 1) are aligned and take one load each; with pairs from column 0 on every source took two
// (update_pair).  Rows 2 .. nr - 3: there a load past an unstored lane's column stays inside its
// plane.  The arithmetic is update_pair's.
template <int STO>
__device__ __forceinline__ void pair_odd(const Consts<float>& c, const Buf<STO>& A, const Buf<STO>& B,
                                         const float* __restrict__ phi, int plane, int kr, int n) {
    const int nz = c.nz, kz0 = 2 * n - (kr & 1), row = kr * nz, rowm = row - nz, rowp = row + nz;
    const bool st0 = kz0 > 0 && kz0 < nz - 1, st1 = kz0 + 1 > 0 && kz0 + 1 < nz - 1;
    if (!st0 && !st1) return;
    const auto* __restrict__ F = A.f;
    const float* __restrict__ G = A.g;
    const auto vec = [&](const auto* p, int o) { return ld2<true>(p, o, o + 1, true); };
    const auto two = [&](const auto* p, int o) { return ld2<true>(p, o, o + 1, false); };
    V2 fh[9], gh[5];
    fh[0] = vec(F, row + kz0);
    fh[1] = two(F + plane, rowm + kz0);
    fh[2] = two(F + 2 * plane, row + kz0 - 1);
    fh[3] = two(F + 3 * plane, rowp + kz0);
    fh[4] = two(F + 4 * plane, row + kz0 + 1);
    fh[5] = vec(F + 5 * plane, rowm + kz0 - 1);
    fh[6] = vec(F + 6 * plane, rowp + kz0 - 1);
    fh[7] = vec(F + 7 * plane, rowp + kz0 + 1);
    fh[8] = vec(F + 8 * plane, rowm + kz0 + 1);
    gh[0] = vec(G, row + kz0);
    gh[1] = two(G + plane, rowm + kz0);
    gh[2] = two(G + 2 * plane, row + kz0 - 1);
    gh[3] = two(G + 3 * plane, rowp + kz0);
    gh[4] = two(G + 4 * plane, row + kz0 + 1);
    const V2 ph = vec(phi, row + kz0);
    const auto qw = [&](int rs, int cs) {
        const int o = (rs == 0 ? rowm : rs == 1 ? row : rowp) + kz0 + cs - 1;
        return ldq2<true>(c.fref, o, o + 1, (rs == 1) == (cs == 1));
    };
    pair_finish<STO, true>(c, B, plane, kr, row, kz0, 1, 5, 8, fh, gh, ph, qw, st0, st1);
}

// Interior pair n, numbered through all rows.
template <int STO, bool VEC>
__device__ __forceinline__ void inner16(const Consts<float>& c, const Buf<STO>& A, const Buf<STO>& B,
                                        const float* __restrict__ phi, int plane, int n) {
    const int P = (c.nz + 1) >> 1, y = n / P, kr = step_row0(c.geometry) + y;
    if (!VEC && !c.periodic && kr >= 2 && kr <= c.nr - 3) {
        pair_odd<STO>(c, A, B, phi, plane, kr, n - y * P);
    } else {
        update_pair<STO, VEC, true>(c, A, B, phi, plane, kr, 1, 2 * (n - y * P));
    }
}

// One step: the blocks of the boundary nodes first.  Against k_bulk_pair and k_wall, BF16, per step:
// 48 x 96 4.5 against 11.0 us, 300 x 601 7.6 against 17.2, 1023 x 2047 38 against 48 (39 with
// pairs from column 0 on), 4096 x 8191 0.53 against 0.60 ms.
template <int STO, bool VEC>
__global__ void __launch_bounds__(BULK_THREADS, 6) k_step16(const Step16 s, int from, int walls) {
    const int wall_blocks = (walls + BULK_THREADS - 1) / BULK_THREADS;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const Buf<STO> A = buf16<STO>(s, from), B = buf16<STO>(s, from ^ 1);
    if ((int)blockIdx.x < wall_blocks) {
        const int n = blockIdx.x * BULK_THREADS + threadIdx.x;
        if (n < walls) wall16<STO>(s.c, A, B, s.phi, s.plane, n);
    } else {
        inner16<STO, VEC>(s.c, A, B, s.phi, (int)s.plane,
                          ((int)blockIdx.x - wall_blocks) * BULK_THREADS + threadIdx.x);
    }
}

// Fields of interior pair n: update_pair's pull and recovery.
template <int STO, bool VEC>
__device__ __forceinline__ void fields_pair16(const Consts<float>& c, const Buf<STO>& A, const float* __restrict__ phi,
                                              int plane, int n, const Fields& o) {
    const int nz = c.nz, P = (nz + 1) >> 1, y = n / P, kr = step_row0(c.geometry) + y, kz = 2 * (n - y * P);
    const bool pz = c.periodic != 0, in1 = kz + 1 < nz;
    const bool st0 = pz || (kz > 0 && kz < nz - 1), st1 = in1 && (pz || kz + 1 < nz - 1);
    if (kr >= c.nr - 1 || (!st0 && !st1)) return;
    const int zc = in1 ? kz + 1 : kz, zm = kz > 0 ? kz - 1 : (pz ? nz - 1 : 0), z0 = in1 ? kz + 1 : (pz ? 0 : nz - 1);
    const int z1 = kz + 2 < nz ? kz + 2 : (pz ? kz + 2 - nz : nz - 1);
    const int row = kr * nz, rowp = row + nz, rowm = kr == 0 ? row : row - nz;   // (pipe axis: mirror image)
    const int p1 = kr == 0 ? 3 : 1, p5 = kr == 0 ? 6 : 5, p8 = kr == 0 ? 7 : 8;
    const auto* __restrict__ F = A.f;
    const float* __restrict__ G = A.g;
    const auto own = [&](const auto* p, int r) { return ld2<true>(p, r + kz, r + zc, VEC); };
    const auto left = [&](const auto* p, int r) { return ld2<true>(p, r + zm, r + kz, false); };
    const auto right = [&](const auto* p, int r) { return ld2<true>(p, r + z0, r + z1, false); };
    V2 fh[9] = {own(F, row), own(F + p1 * plane, rowm), left(F + 2 * plane, row), own(F + 3 * plane, rowp),
                right(F + 4 * plane, row), left(F + p5 * plane, rowm), left(F + 6 * plane, rowp),
                right(F + 7 * plane, rowp), right(F + p8 * plane, rowm)};
    V2 gh[5] = {own(G, row), own(G + p1 * plane, rowm), left(G + 2 * plane, row), own(G + 3 * plane, rowp),
                right(G + 4 * plane, row)};
    const V2 ph = own(phi, row);
    const Q2 q0 = ldq2<true>(c.fref, row + kz, row + zc, VEC);
    const V2 R = q0.R;
    const auto add = [&](int r, int a, int b, bool vec, int i0, int s0, int i1, int s1, int i2, int s2) {
        const Q2 q = ldq2<true>(c.fref, r + a, r + b, vec);
        if (i0 >= 0) fh[i0] += fref_delta2(s0, q);
        if (i1 >= 0) fh[i1] += fref_delta2(s1, q);
        if (i2 >= 0) gh[i2] += 0.1f * (q.R - R);
    };
    fh[0] += fref_delta2(0, q0);
    add(row, zm, kz, false, 2, 2, -1, 0, 2, 0);
    add(row, z0, z1, false, 4, 4, -1, 0, 4, 0);
    add(rowm, kz, zc, VEC, 1, p1, -1, 0, 1, 0);
    add(rowm, zm, kz, false, 5, p5, -1, 0, -1, 0);
    add(rowm, z0, z1, false, 8, p8, -1, 0, -1, 0);
    add(rowp, kz, zc, VEC, 3, 3, -1, 0, 3, 0);
    add(rowp, zm, kz, false, 6, 6, -1, 0, -1, 0);
    add(rowp, z0, z1, false, 7, 7, -1, 0, -1, 0);
    V2 lin, nl, iph, m0, rho, ur, uz, dT;
    porous2(c, ph, lin, nl, iph);
    recover2(c, row_consts(c, kr), ph, lin, nl, fh, gh, R, m0, rho, ur, uz, dT);
    put_pair(o, row + kz, st0, st1, rho, ur, uz, (c.T0 + R) + dT);
}
template <int STO, bool VEC>
__global__ void __launch_bounds__(BULK_THREADS, 8) k_fields16(const Step16 s, int which, int walls, const Fields o) {
    const int wall_blocks = (walls + BULK_THREADS - 1) / BULK_THREADS;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const Buf<STO> A = buf16<STO>(s, which);
    if ((int)blockIdx.x < wall_blocks) {
        const int n = blockIdx.x * BULK_THREADS + threadIdx.x;
        if (n >= walls) return;
        const Consts<float>& c = s.c;
        int kr, kz;
        wall_node(c.geometry, c.nr, c.nz, n, kr, kz);
        float fh[9], gh[5], m0, rho, ur, uz, dT, ref;
        wall_state<STO, float, LAY_N, true>(c, A, s.phi, s.plane, node_class(c.geometry, c.nr, c.nz, kr, kz), kr, kz, fh, gh, m0, rho, ur,
                               uz, dT, ref);
        const float v[4] = {rho, ur, uz, (c.T0 + ref) + dT};
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (o.p[k]) o.p[k][kr * c.nz + kz] = v[k];
    } else {
        fields_pair16<STO, VEC>(s.c, A, s.phi, (int)s.plane, ((int)blockIdx.x - wall_blocks) * BULK_THREADS + threadIdx.x, o);
    }
}

// The same for the instances of a batch, whose constants are read from shared memory.  16 instances
// of 64 to 160 rows (450 k nodes, FP16): 10.2 us per step (19.0 with staged tiles and the forked wall
// kernel); 16 of 200 to 400 (3.6 M nodes, BF16) 68 against 76; 64 of 64 to 512 (12.2 M nodes) 232
// against 231, where the staged tiles serve.  The staged tiles with the boundary nodes in their
// launch: 234.  Six blocks per SM, for even nz (five / six / seven: 16 of 200 x 400 25.8 / 25.2 / 26.7 us,
// 32 of 300 x 600 113 / 109 / 115).  The odd-nz form spills 196 bytes at six (even: 40) and would do best
// with five: 16 of 100 x 201 8.7 / 9.9 / 11.2 us, 16 of 200 x 401 27.4 / 31.4 / 33.4, 32 of 300 x 601
// 116 / 130 / 137 (staged tiles' k_batch_bulk and the wall kernel before: 35.8 for 16 of 200 x 401).
template <int STO, bool VEC>
__global__ void __launch_bounds__(BULK_THREADS, 6) k_batch_step16(const Step16* __restrict__ inst,
                                                                  const int2* __restrict__ blocks, int from) {
    __shared__ Step16 s;
    const int2 b = blocks[blockIdx.x];   // the lists and constants are not written by a launch
    for (int w = threadIdx.x; w < (int)(sizeof(Step16) / sizeof(int)); w += BULK_THREADS)
        reinterpret_cast<int*>(&s)[w] = reinterpret_cast<const int*>(inst + (b.x >> 1))[w];
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const Buf<STO> A = buf16<STO>(s, from), B = buf16<STO>(s, from ^ 1);
    const int n = b.y + threadIdx.x;
    if (b.x & 1) {
        if (n < step_walls(s.c.geometry, s.c.nr, s.c.nz)) {
            const Consts<float> c = s.c;
            wall16<STO>(c, A, B, s.phi, s.plane, n);
        }
    } else {
        inner16<STO, VEC>(s.c, A, B, s.phi, (int)s.plane, n);
    }
}
namespace lbm {

cudaError_t launch16(int storage, const Step16& s, int from, cudaStream_t stream) {
    const Consts<float>& c = s.c;
    const int walls = step_walls(c.geometry, c.nr, c.nz), wb = (walls + BULK_THREADS - 1) / BULK_THREADS;
    const int pairs = step_pairs(c.geometry, c.nr, c.nz), pb = (pairs + BULK_THREADS - 1) / BULK_THREADS;
    const auto k = storage == LBM_F16 ? (c.nz & 1 ? k_step16<LBM_F16, false> : k_step16<LBM_F16, true>)
                                      : (c.nz & 1 ? k_step16<LBM_BF16, false> : k_step16<LBM_BF16, true>);
    return launch_dependent(k, (unsigned)(wb + pb), BULK_THREADS, 0, stream, s, from, walls);
}

Blocks16 blocks16(const std::vector<lbm_params>& p, const std::vector<int>& act) {
    Blocks16 out;
    for (int kind = 1; kind >= 0; --kind)
        for (int i : act) {
            const int n = kind ? step_walls(p[i].geometry, p[i].nr, p[i].nz) : step_pairs(p[i].geometry, p[i].nr, p[i].nz);
            for (int k = 0; k < n; k += BULK_THREADS) ((p[i].nz & 1) ? out.odd : out.even).push_back(make_int2(2 * i + kind, k));
        }
    return out;
}

cudaError_t launch_batch16(int storage, const Step16* inst, const int2* blocks, int n, bool odd_nz, int from,
                           cudaStream_t stream) {
    const auto k = storage == LBM_F16 ? (odd_nz ? k_batch_step16<LBM_F16, false> : k_batch_step16<LBM_F16, true>)
                                      : (odd_nz ? k_batch_step16<LBM_BF16, false> : k_batch_step16<LBM_BF16, true>);
    return launch_dependent(k, (unsigned)n, BULK_THREADS, 0, stream, inst, blocks, from);
}

cudaError_t launch_fields16(int storage, const Step16& s, int which, float* rho, float* ur, float* uz, float* T,
                            cudaStream_t stream) {
    const Consts<float>& c = s.c;
    const int walls = step_walls(c.geometry, c.nr, c.nz), pairs = step_pairs(c.geometry, c.nr, c.nz);
    const unsigned blocks = (walls + BULK_THREADS - 1) / BULK_THREADS + (pairs + BULK_THREADS - 1) / BULK_THREADS;
    const auto k = storage == LBM_F16 ? (c.nz & 1 ? k_fields16<LBM_F16, false> : k_fields16<LBM_F16, true>)
                                      : (c.nz & 1 ? k_fields16<LBM_BF16, false> : k_fields16<LBM_BF16, true>);
    return launch_dependent(k, blocks, BULK_THREADS, 0, stream, s, which, walls, fields_of(c.nz, rho, ur, uz, T));
}

}  // namespace lbm
