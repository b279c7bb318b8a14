// lbm_nodes.cuh -- storage of the state and the node updates that the kernels of lbm.cu and
// lbm_16.cu share: where populations are kept and how they are pulled and stored, the boundary
// rebuild, the scalar column update, the packed pair update and the staged block of 16-bit
// storage.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "../../include/lbm.h"
#include "lbm_pair.cuh"
#include "lbm_physics.cuh"

using namespace lbm;

// ------------------------------------------------------------ storage types --
// Flow populations in the storage type; temperature populations always FP32 (in
// 16 bits the per-step change of g - wT T0, of order 0.05, falls below the format's
// resolution and the temperature field stagnates); porosity always FP32 (in FP16 its
// half-ulp, 2.4e-4 relative near 0.7, moves the Darcy drag of Eq. 8 by about 2e-3).
//
// Loads.  DEP: the kernel is launched dependently (lbm_dependent.h), so it is resident while the
// launch before it may still write the state, the references or the porosity; only an ordinary load
// stays behind its wait.  The read-only load (__ldg) wants data that no one writes during the whole
// life of the kernel.
template <bool DEP, class T> __device__ __forceinline__ T ld1(const T* p) {
    if constexpr (DEP) return *p;
    else return __ldg(p);
}
template <bool DEP = false> __device__ __forceinline__ float ldv(const float* p) { return ld1<DEP>(p); }
template <bool DEP = false> __device__ __forceinline__ float ldv(const __half* p) { return __half2float(ld1<DEP>(p)); }
template <bool DEP = false> __device__ __forceinline__ float ldv(const __nv_bfloat16* p) {
    return __bfloat162float(ld1<DEP>(p));
}
__device__ __forceinline__ void stv(float* p, float v) { *p = v; }
__device__ __forceinline__ void stv(__half* p, float v) { *p = __float2half_rn(v); }
__device__ __forceinline__ void stv(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

template <int STO> struct St;
template <> struct St<LBM_F32> { using TF = float; using TG = float; using P = float; };
template <> struct St<LBM_F16> { using TF = __half; using TG = float; using P = float; };
template <> struct St<LBM_BF16> { using TF = __nv_bfloat16; using TG = float; using P = float; };

// One state buffer: nine flow planes then five temperature planes.
template <int STO> struct Buf {
    typename St<STO>::TF* f;
    typename St<STO>::TG* g;
};

static size_t f_size(int sto) { return sto == LBM_F32 ? 4 : 2; }
static size_t g_size(int) { return 4; }
static size_t phi_size(int) { return 4; }
static size_t state_bytes(int sto, int64_t plane) { return (size_t)plane * (9 * f_size(sto) + 5 * g_size(sto)); }

constexpr int BULK_THREADS = 128;
#ifndef LBM_BULK_RPT
#define LBM_BULK_RPT 4
#endif
constexpr int BULK_RPT = LBM_BULK_RPT;  // rows per thread of the bulk kernel (32-bit indexing)
#ifndef LBM_BULK_RPT_MIN_BLOCKS
#define LBM_BULK_RPT_MIN_BLOCKS 16
#endif
// BULK_RPT rows per thread only where the grid keeps at least this many blocks per SM
constexpr int BULK_RPT_MIN_BLOCKS = LBM_BULK_RPT_MIN_BLOCKS;

// ------------------------------------------------------------- layouts --
// Where the post-collision population i of node y is kept between steps:
//   LAY_N  two state buffers (A/B): slot i at y of the buffer last written;
//   LAY_S  one buffer (in place), after an even number of steps: slot opp(i) at y;
//   LAY_L  one buffer, after an odd number of steps: slot i at y + e_i (z wraps when
//          periodic; populations leaving through the pipe axis are kept where the axis
//          row's pull reads them: f+_3(0, z) at (1, (0, z)), f+_6(0, z) at (5, (0, z + 1)),
//          f+_7(0, z) at (8, (0, z - 1)); other populations leaving the domain are dropped).
// A step of the in-place scheme reads S and writes L, or reads L and writes S: every
// location a node reads is one it writes and no other node touches it, so one buffer
// suffices.  The same layouts hold for the five temperature populations.
enum { LAY_N = 0, LAY_S = 1, LAY_L = 2 };
__host__ __device__ constexpr int opp9(int i) { return i == 0 ? 0 : i < 5 ? ((i + 1) & 3) + 1 : ((i - 3) & 3) + 5; }

// ------------------------------------------------------------- pull (Eq. 22) --
// Sources of the pulled populations at (kr, kz): the node src[i] whose post-collision
// population sp[i] streams into population i, i.e. (kr - e_ir) nz + (kz - e_iz), and in the
// pipe's axis row for the e_r = +1 populations the node's mirror image (population
// mirror(i) of row 0); and, for layout LAY, where that value is kept: node loc[i], slot
// lp[i].  Periodic z wraps.
template <int LAY, typename R, typename I>
__device__ __forceinline__ void pull_sources(const Consts<R>& c, int kr, int kz, I* src, int* sp, I* loc, int* lp) {
    const bool pz = c.periodic != 0;
    const int zm = (pz && kz == 0) ? c.nz - 1 : kz - 1;       // source column for e_z = +1
    const int zp = (pz && kz == c.nz - 1) ? 0 : kz + 1;       // source column for e_z = -1
    const I row = (I)kr * c.nz;
    const I rowm = row - c.nz, rowp = row + c.nz;
    const bool axis = (kr == 0);                              // reached only in the pipe
    src[0] = row + kz;        sp[0] = 0;
    src[1] = (axis ? row : rowm) + kz;  sp[1] = axis ? 3 : 1;
    src[2] = row + zm;        sp[2] = 2;
    src[3] = rowp + kz;       sp[3] = 3;
    src[4] = row + zp;        sp[4] = 4;
    src[5] = (axis ? row : rowm) + zm;  sp[5] = axis ? 6 : 5;
    src[6] = rowp + zm;       sp[6] = 6;
    src[7] = rowp + zp;       sp[7] = 7;
    src[8] = (axis ? row : rowm) + zp;  sp[8] = axis ? 7 : 8;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        loc[i] = LAY == LAY_L ? row + kz : src[i];
        lp[i] = LAY == LAY_N ? sp[i] : LAY == LAY_S ? opp9(sp[i]) : i;
    }
}

// Where node (kr, kz) keeps its post-collision population i in layout LAY (false: dropped).
template <int LAY, typename R, typename I>
__device__ __forceinline__ bool own_slot(const Consts<R>& c, int kr, int kz, int i, I& node, int& slot) {
    if (LAY != LAY_L) {
        node = (I)kr * c.nz + kz;
        slot = LAY == LAY_N ? i : opp9(i);
        return true;
    }
    int r = kr + ex9(i), z = kz + ez9(i);
    slot = i;
    if (r < 0) {   // leaving through row 0: kept only on the pipe axis, as its mirror image
        if (c.geometry != PIPE_PERIODIC_Z && c.geometry != PIPE_INFLOW) return false;
        r = 0;         // the mirror image keeps the z motion: (0, z + e_iz)
        slot = i == 3 ? 1 : i == 6 ? 5 : 8;
    }
    if (r >= c.nr) return false;
    if (z < 0 || z >= c.nz) {
        if (!c.periodic) return false;
        z = z < 0 ? z + c.nz : z - c.nz;
    }
    node = (I)r * c.nz + z;
    return true;
}

// Flow populations stored against a per-node reference (16-bit storage, see fref_delta).
template <int STO> __host__ __device__ constexpr bool has_fref() { return STO != LBM_F32; }

// Pre-collision deviations at (kr, kz) from the post-collision state A in layout LAY: a
// plain copy of ft_i(x - e_i) (see lbm_physics.cuh), plus, with 16-bit storage, the
// reference part D_pop(Q(source)) of the value the source node stored.  src receives the
// source nodes (for the temperature reference).
template <int STO, int LAY, bool DEP, typename R, typename I>
__device__ __forceinline__ void pull_raw(const Consts<R>& c, const Buf<STO>& A, I plane, int kr, int kz, R* fh,
                                         R* gh, I* src) {
    I loc[9];
    int sp[9], lp[9];
    pull_sources<LAY, R, I>(c, kr, kz, src, sp, loc, lp);
    const auto* __restrict__ F = A.f;
    const auto* __restrict__ G = A.g;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        float v = ldv<DEP>(F + lp[i] * plane + loc[i]);
        if constexpr (has_fref<STO>()) v += fref_delta(sp[i], fref_unpack(c.fref[src[i]]));
        fh[i] = R(v);
    }
#pragma unroll
    for (int i = 0; i < 5; ++i) gh[i] = R(ldv<DEP>(G + lp[i] * plane + loc[i]));
}

// Re-reference pulled thermal deviations to the node's R(x): gh_i += wT_i (R(x - e_i) - R(x))
// with r0 = R(x) and rm, zm, rp, zp the offsets of the sources of g_1 .. g_4.
template <typename R>
__device__ __forceinline__ void reref(R* gh, R r0, R rm, R zm, R rp, R zp) {
    gh[1] += R(0.1) * (rm - r0);
    gh[2] += R(0.1) * (zm - r0);
    gh[3] += R(0.1) * (rp - r0);
    gh[4] += R(0.1) * (zp - r0);
}

// Every storage type keeps the temperature reference R(x): the FP32 temperature populations
// stored against T0 alone would carry deviations of size |T - T0|, on which FP32 arithmetic
// biases the thermal update and freezes slow modes short of their fixed point.
template <int STO> __host__ __device__ constexpr bool has_ref() { return true; }

// R(x) of node n: its own FP16 plane with FP32 storage, the fourth FP16 of the node's
// reference word with 16-bit storage.
template <int STO, typename R, typename I>
__device__ __forceinline__ float tref_at(const Consts<R>& c, I n) {
    if constexpr (has_fref<STO>()) {
        const uint32_t w = c.fref[n].y;
        return __high2float(*reinterpret_cast<const __half2*>(&w));
    } else {
        return __half2float(c.tref[n]);
    }
}

// Pull (Eq. 22) from layout LAY with the thermal deviations re-referenced to R(x), which
// *rref receives (on the pipe axis row g_1 comes from the node's own mirror image).
template <int STO, typename R, typename I = int64_t, int LAY = LAY_N, bool DEP = false>
__device__ __forceinline__ void pull(const Consts<R>& c, const Buf<STO>& A, I plane, int kr, int kz, R* fh, R* gh,
                                     R& rref) {
    I src[9];
    pull_raw<STO, LAY, DEP, R, I>(c, A, plane, kr, kz, fh, gh, src);
    rref = R(tref_at<STO>(c, (I)kr * c.nz + kz));
    reref(gh, rref, R(tref_at<STO>(c, src[1])), R(tref_at<STO>(c, src[2])), R(tref_at<STO>(c, src[3])),
          R(tref_at<STO>(c, src[4])));
}

// Store the post-collision deviations of node (kr, kz) = n in layout LAY (16-bit storage:
// against the node's own flow reference Q(n)).
template <int STO, typename R, typename I = int64_t, int LAY = LAY_N>
__device__ __forceinline__ void store(const Consts<float>& c, const Buf<STO>& B, I plane, int kr, int kz, I n,
                                      const R* fh, const R* gh) {
    Qf q;
    if constexpr (has_fref<STO>()) q = fref_unpack(c.fref[n]);
    if constexpr (LAY == LAY_N) {
        // two buffers: the nine flow planes, then the five temperature planes (measured 7 %
        // faster than interleaved)
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            float v = float(fh[i]);
            if constexpr (has_fref<STO>()) v -= fref_delta(i, q);
            stv(B.f + i * plane + n, v);
        }
#pragma unroll
        for (int i = 0; i < 5; ++i) stv(B.g + i * plane + n, float(gh[i]));
    } else {
        // in place: f_i and g_i of one direction together, at the location own_slot gives
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            I m;
            int slot;
            if (!own_slot<LAY, float, I>(c, kr, kz, i, m, slot)) continue;
            float v = float(fh[i]);
            if constexpr (has_fref<STO>()) v -= fref_delta(i, q);
            stv(B.f + slot * plane + m, v);
            if (i < 5) stv(B.g + slot * plane + m, float(gh[i]));
        }
    }
}

// Boundary node state: rebuild (Sec. 4, ref. [47]) from the interior neighbour, then
// rho from Eq. 26.  Walls: u_b = 0, rho_b = rho_f, T_b = T_hot (inner), T_cold (outer),
// T_f (adiabatic top and bottom).  Pipe inlet: u_b = (0, u_in), rho_b = rho_f, T_b = T_hot;
// outlet: u_b = u_f, T_b = T_f, rho_b = 1 (zero gradient of u and T, density held).
template <int STO, typename R, int LAY = LAY_N, bool DEP = false>
__device__ __forceinline__ void wall_state(const Consts<R>& c, const Buf<STO> A,
                                           const typename St<STO>::P* __restrict__ phi, int64_t plane, int cls,
                                           int kr, int kz, R* fh, R* gh, R& m0, R& rho, R& urb, R& uzb, R& dTb,
                                           R& refb) {
    int fr, fz;
    fluid_neighbour(c.geometry, c.nr, c.nz, cls, kr, kz, fr, fz);
    R fhf[9], ghf[5], reff;
    pull<STO, R, int64_t, LAY, DEP>(c, A, plane, fr, fz, fhf, ghf, reff);
    const R rf = c.r0 + R(fr), rb = c.r0 + R(kr);
    const R phif = R(ldv<DEP>(phi + (int64_t)fr * c.nz + fz));
    R m0f, rhof, urf, uzf, dTf, lin, nl, ipf;
    porous(c, phif, lin, nl, ipf);
    recover(c, rf, rcp_acc(rf), phif, lin, nl, fhf, ghf, reff, m0f, rhof, urf, uzf, dTf);
    R drhob = m0f * rcp_acc(rf), rhob = rhof;
    urb = R(0);
    uzb = R(0);
    R ipb = R(1);
    if (cls == INLET) {
        uzb = c.u_in;
    } else if (cls == OUTLET) {
        urb = urf;
        uzb = uzf;
        drhob = R(0);
        rhob = R(1);
    }
    if (cls >= INLET) ipb = rcp_acc(R(ldv<DEP>(phi + (int64_t)kr * c.nz + kz)));
    rebuild_flow(rb, rf, ipb, ipf, drhob, rhob, urb, uzb, m0f, rhof, urf, uzf, fhf, fh);
    // deviations relative to this boundary node's own reference R_b
    refb = R(tref_at<STO>(c, (int64_t)kr * c.nz + kz));
    dTb = (cls == WALL_IN || cls == INLET) ? (c.T_hot - c.T0) - refb
          : cls == WALL_OUT                 ? (c.T_cold - c.T0) - refb
                                            : (dTf + reff) - refb;
    if (cls == WALL_IN && c.heater) {
        // Sec. 4.4: q' = -k dT/dr on the heater, dT/dr = 0 on the rest of the inner wall;
        // (-3 T_b + 4 T_1 - T_2) / 2 = -q'/k with the next two nodes inward (T_1 = T_f);
        // corners (diagonal neighbour) take T_f
        if (fz == kz) {
            R f2[9], g2[5], ref2;
            pull<STO, R, int64_t, LAY, DEP>(c, A, plane, 2, kz, f2, g2, ref2);
            const R T1 = (c.T0 + reff) + dTf;
            const R T2 = (c.T0 + ref2) + (((g2[0] + g2[1]) + (g2[2] + g2[3])) + g2[4]);
            const R G = (kz >= c.hz0 && kz <= c.hz1) ? c.hG : R(0);
            dTb = (R(4) * T1 - T2 + R(2) * G) * R(1.0 / 3.0) - (c.T0 + refb);
        } else {
            dTb = (dTf + reff) - refb;
        }
    }
    rebuild_thermal(c.T0 + reff, dTf, c.T0 + refb, dTb, urb, uzb, urf, uzf, ghf, gh);
    m0 = ((fh[0] + fh[1]) + (fh[2] + fh[3])) + ((fh[4] + fh[5]) + (fh[6] + fh[7])) + fh[8];
    rho = R(1) + m0 * rcp_acc(rb);
}

// Boundary node t -> (kr, kz): inner wall (annulus), outer wall, then bottom and top
// without the corners (closed annulus).  Pipe with inlet: inlet row, outlet row, then
// the wall without the corners.
__device__ __forceinline__ void wall_node(int geometry, int nr, int nz, int t, int& kr, int& kz) {
    if (geometry == PIPE_INFLOW) {
        if (t < nr) { kr = t; kz = 0; return; }
        t -= nr;
        if (t < nr) { kr = t; kz = nz - 1; return; }
        t -= nr;
        kr = nr - 1;
        kz = 1 + t;
        return;
    }
    if (geometry != PIPE_PERIODIC_Z) {
        if (t < nz) { kr = 0; kz = t; return; }
        t -= nz;
    }
    if (t < nz) { kr = nr - 1; kz = t; return; }
    t -= nz;
    if (t < nr - 2) { kr = 1 + t; kz = 0; return; }
    t -= nr - 2;
    kr = 1 + t;
    kz = nz - 1;
}

static int wall_count(int geometry, int nr, int nz) {
    if (geometry == ANNULUS) return 2 * nz + 2 * (nr - 2);
    if (geometry == ANNULUS_PERIODIC_Z) return 2 * nz;
    if (geometry == PIPE_INFLOW) return 2 * nr + nz - 2;
    return nz;
}

// ------------------------------------------------------------------ kernels --
// Update `rows` consecutive non-wall nodes of column kz from row kr0 on (rows past the
// last row are skipped); shared by the single-problem and the batched bulk kernels.
// I: index type.
template <int STO, typename I, int LIN = LAY_N, int LOUT = LAY_N>
__device__ __forceinline__ void update_column(const Consts<float>& c, const Buf<STO>& A, const Buf<STO>& B,
                                              const typename St<STO>::P* __restrict__ phi, I plane, int kr0,
                                              int rows, int kz) {
    // node_class split into its column and row parts: the end columns are boundary
    // nodes unless z is periodic; row nr - 1 is a wall, row 0 too unless it is a pipe axis
    const bool zwall = !c.periodic && (kz == 0 || kz == c.nz - 1);
    const bool row0_wall = c.geometry == ANNULUS || c.geometry == ANNULUS_PERIODIC_Z;
#pragma unroll 1
    for (int j = 0; j < rows; ++j) {
        const int kr = kr0 + j;
        if (kr >= c.nr) break;
        if (zwall || kr == c.nr - 1 || (kr == 0 && row0_wall)) continue;
        float fh[9], gh[5], ref;
        pull<STO, float, I, LIN>(c, A, plane, kr, kz, fh, gh, ref);
        const I n = (I)kr * c.nz + kz;
        const float r = c.r0 + float(kr), inv_r = rcp_acc(r);
        const float ph = ldv(phi + n);
        float m0, rho, ur, uz, dT, lin, nl, iph;
        porous(c, ph, lin, nl, iph);
        recover(c, r, inv_r, ph, lin, nl, fh, gh, ref, m0, rho, ur, uz, dT);
        collide(c, r, inv_r, ph, lin, nl, iph, fh, gh, ref, m0, rho, ur, uz, dT);
        store<STO, float, I, LOUT>(c, B, plane, kr, kz, n, fh, gh);
    }
}

// ------------------------------------------- packed pair update (16-bit storage) --
// Two z-adjacent nodes (kz0, kz0 + 1) per thread, their arithmetic on the packed FP32
// instructions of lbm_pair.cuh.  Loads of the node's own columns are single vector loads
// when the row's first element index is even (VEC: nz even, kz0 even); the shifted
// columns of the e_z = +-1 populations are two scalar loads.  Flow populations carry the
// flow reference: the pull adds D_pop(Q(source)), the store subtracts D_i(Q(own)).
template <bool DEP = false> __device__ __forceinline__ V2 ld2(const __half* p, int a, int b, bool vec) {
    if (vec) return {__half22float2(ld1<DEP>(reinterpret_cast<const __half2*>(p + a)))};
    return v2(ldv<DEP>(p + a), ldv<DEP>(p + b));
}
template <bool DEP = false> __device__ __forceinline__ V2 ld2(const __nv_bfloat16* p, int a, int b, bool vec) {
    if (vec) return {__bfloat1622float2(ld1<DEP>(reinterpret_cast<const __nv_bfloat162*>(p + a)))};
    return v2(ldv<DEP>(p + a), ldv<DEP>(p + b));
}
template <bool DEP = false> __device__ __forceinline__ V2 ld2(const float* p, int a, int b, bool vec) {
    if (vec) return {ld1<DEP>(reinterpret_cast<const float2*>(p + a))};
    return v2(ldv<DEP>(p + a), ldv<DEP>(p + b));
}
template <bool DEP = false> __device__ __forceinline__ Q2 ldq2(const uint2* q, int a, int b, bool vec) {
    uint2 ua, ub;
    if (vec) {
        const uint4 u = ld1<DEP>(reinterpret_cast<const uint4*>(q + a));
        ua = make_uint2(u.x, u.y);
        ub = make_uint2(u.z, u.w);
    } else {
        ua = ld1<DEP>(q + a);
        ub = ld1<DEP>(q + b);
    }
    const Qf x = fref_unpack(ua), y = fref_unpack(ub);
    return {v2(x.A, y.A), v2(x.Jr, y.Jr), v2(x.Jz, y.Jz), v2(x.R, y.R)};
}

__device__ __forceinline__ void st2(__half* p, int a, V2 v, bool s0, bool s1, bool vec) {
    const __half2 h = __floats2half2_rn(v.v.x, v.v.y);
    if (vec && s0 && s1) {
        *reinterpret_cast<__half2*>(p + a) = h;
    } else {
        if (s0) p[a] = __low2half(h);
        if (s1) p[a + 1] = __high2half(h);
    }
}
__device__ __forceinline__ void st2(__nv_bfloat16* p, int a, V2 v, bool s0, bool s1, bool vec) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v.v.x, v.v.y);
    if (vec && s0 && s1) {
        *reinterpret_cast<__nv_bfloat162*>(p + a) = h;
    } else {
        if (s0) p[a] = __low2bfloat16(h);
        if (s1) p[a + 1] = __high2bfloat16(h);
    }
}
__device__ __forceinline__ void st2(float* p, int a, V2 v, bool s0, bool s1, bool vec) {
    if (vec && s0 && s1) {
        *reinterpret_cast<float2*>(p + a) = v.v;
    } else {
        if (s0) p[a] = v.v.x;
        if (s1) p[a + 1] = v.v.y;
    }
}

// The rest of one row of a column pair once its sources are loaded: the flow reference
// added back (D_pop of each source's word; g_1 .. g_4 re-expressed against the node's own
// temperature reference), the recovery and collision, and the store with the own word's
// D_i removed.  qw(rs, cs): the two reference words of the sources in row kr - 1 + rs and
// columns (kz0 - 1, kz0), (kz0, kz0 + 1) or (kz0 + 1, kz0 + 2) for cs = 0, 1, 2.
template <int STO, bool VEC, class QW>
__device__ __forceinline__ void pair_finish(const Consts<float>& c, const Buf<STO>& B, int plane, int kr, int row,
                                            int kz0, int p1, int p5, int p8, V2 (&fh)[9], V2 (&gh)[5], V2 ph,
                                            const QW& qw, bool st0, bool st1) {
    // the reference words of the sources: the flow part D_pop of the pulled values and,
    // in their fourth slot, the temperature references R that re-express g_1 .. g_4
    // against the node's own R(x)
    const Q2 q0o = qw(1, 1);
    const V2 rref = q0o.R;
    {
        const Q2 qmo = qw(0, 1), qml = qw(0, 0), qmr = qw(0, 2);
        fh[1] += fref_delta2(p1, qmo);
        fh[5] += fref_delta2(p5, qml);
        fh[8] += fref_delta2(p8, qmr);
        gh[1] += 0.1f * (qmo.R - rref);
        const Q2 q0l = qw(1, 0), q0r = qw(1, 2);
        fh[0] += fref_delta2(0, q0o);
        fh[2] += fref_delta2(2, q0l);
        fh[4] += fref_delta2(4, q0r);
        gh[2] += 0.1f * (q0l.R - rref);
        gh[4] += 0.1f * (q0r.R - rref);
        const Q2 qpo = qw(2, 1), qpl = qw(2, 0), qpr = qw(2, 2);
        fh[3] += fref_delta2(3, qpo);
        fh[6] += fref_delta2(6, qpl);
        fh[7] += fref_delta2(7, qpr);
        gh[3] += 0.1f * (qpo.R - rref);
    }
    const RowC q = row_consts(c, kr);
    V2 lin, nl, iph, m0, rho, ur, uz, dT;
    porous2(c, ph, lin, nl, iph);
    recover2(c, q, ph, lin, nl, fh, gh, rref, m0, rho, ur, uz, dT);
    collide2(c, q, ph, lin, nl, iph, fh, gh, rref, m0, rho, ur, uz, dT);
    auto* __restrict__ Fo = B.f;
    float* __restrict__ Go = B.g;
#pragma unroll
    for (int i = 0; i < 9; ++i) fh[i] = fh[i] - fref_delta2(i, q0o);
    if (VEC && st0 && st1) {   // both lanes stored, aligned: one vector store per population
#pragma unroll
        for (int i = 0; i < 9; ++i) st2(Fo + i * plane, row + kz0, fh[i], true, true, true);
#pragma unroll
        for (int i = 0; i < 5; ++i) st2(Go + i * plane, row + kz0, gh[i], true, true, true);
    } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) st2(Fo + i * plane, row + kz0, fh[i], st0, st1, false);
#pragma unroll
        for (int i = 0; i < 5; ++i) st2(Go + i * plane, row + kz0, gh[i], st0, st1, false);
    }
}

// Update rows kr0 .. kr0 + rows - 1 (non-wall rows below nr) of the column pair starting
// at the even column kz0.  VEC: nz is even, so every row's first element index is even
// and the own-column pairs are aligned for vector loads and stores.
template <int STO, bool VEC, bool DEP = false>
__device__ __forceinline__ void update_pair(const Consts<float>& c, const Buf<STO>& A, const Buf<STO>& B,
                                            const float* __restrict__ phi, int plane, int kr0, int rows, int kz0) {
    static_assert(has_fref<STO>(), "the packed pair update serves 16-bit storage");
    const int nz = c.nz;
    const bool pz = c.periodic != 0;
    // a lane past the last column, or on the end column of a closed geometry (a boundary
    // node), computes on clamped indices and is not stored
    const bool in1 = kz0 + 1 < nz;
    const bool st0 = pz || (kz0 > 0 && kz0 < nz - 1);   // (kz0 = nz - 1 when nz is odd)
    const bool st1 = in1 && (pz || kz0 + 1 < nz - 1);
    if (!st0 && !st1) return;
    const int zc1 = in1 ? kz0 + 1 : kz0;
    const int zm0 = kz0 > 0 ? kz0 - 1 : (pz ? nz - 1 : 0);          // e_z = +1 source, lane 0
    const int zp0 = in1 ? kz0 + 1 : (pz ? 0 : nz - 1);              // e_z = -1 source, lane 0
    const int zp1 = kz0 + 2 < nz ? kz0 + 2 : (pz ? kz0 + 2 - nz : nz - 1);   // e_z = -1, lane 1
    const bool row0_wall = c.geometry == ANNULUS || c.geometry == ANNULUS_PERIODIC_Z;
    const auto* __restrict__ F = A.f;
    const float* __restrict__ G = A.g;
    const uint2* __restrict__ Qp = c.fref;
#pragma unroll 1
    for (int j = 0; j < rows; ++j) {
        const int kr = kr0 + j;
        if (kr >= c.nr) break;
        if (kr == c.nr - 1 || (kr == 0 && row0_wall)) continue;
        const bool axis = kr == 0;   // pipe axis row: e_r = +1 sources are the mirror image
        const int row = kr * nz, rowp = row + nz, rowm = axis ? row : row - nz;
        const int p1 = axis ? 3 : 1, p5 = axis ? 6 : 5, p8 = axis ? 7 : 8;
        // own (kz0, zc1), left (zm0, kz0) and right (zp0, zp1) columns of a row
        V2 fh[9], gh[5];
        fh[0] = ld2<DEP>(F, row + kz0, row + zc1, VEC);
        fh[1] = ld2<DEP>(F + p1 * plane, rowm + kz0, rowm + zc1, VEC);
        fh[2] = ld2<DEP>(F + 2 * plane, row + zm0, row + kz0, false);
        fh[3] = ld2<DEP>(F + 3 * plane, rowp + kz0, rowp + zc1, VEC);
        fh[4] = ld2<DEP>(F + 4 * plane, row + zp0, row + zp1, false);
        fh[5] = ld2<DEP>(F + p5 * plane, rowm + zm0, rowm + kz0, false);
        fh[6] = ld2<DEP>(F + 6 * plane, rowp + zm0, rowp + kz0, false);
        fh[7] = ld2<DEP>(F + 7 * plane, rowp + zp0, rowp + zp1, false);
        fh[8] = ld2<DEP>(F + p8 * plane, rowm + zp0, rowm + zp1, false);
        gh[0] = ld2<DEP>(G, row + kz0, row + zc1, VEC);
        gh[1] = ld2<DEP>(G + p1 * plane, rowm + kz0, rowm + zc1, VEC);
        gh[2] = ld2<DEP>(G + 2 * plane, row + zm0, row + kz0, false);
        gh[3] = ld2<DEP>(G + 3 * plane, rowp + kz0, rowp + zc1, VEC);
        gh[4] = ld2<DEP>(G + 4 * plane, row + zp0, row + zp1, false);
        const V2 ph = ld2<DEP>(phi, row + kz0, row + zc1, VEC);
        const auto qw = [&](int rs, int cs) {   // words of row kr - 1 + rs, columns left / own / right
            const int r = rs == 0 ? rowm : (rs == 1 ? row : rowp);
            if (cs == 1) return ldq2<DEP>(Qp, r + kz0, r + zc1, VEC);
            if (cs == 0) return ldq2<DEP>(Qp, r + zm0, r + kz0, false);
            return ldq2<DEP>(Qp, r + zp0, r + zp1, false);
        };
        pair_finish<STO, VEC>(c, B, plane, kr, row, kz0, p1, p5, p8, fh, gh, ph, qw, st0, st1);
    }
}

// Reference word of a node from its post-collision deviations d_i = f+_i - rest_i
// (A = sum d_i, J = sum e_i d_i) and its temperature reference R: each rounded to FP16
// after clamping to its range (a clamped or otherwise inexact reference only stores
// larger values).
__device__ __forceinline__ uint2 fref_make(float A, float Jr, float Jz, __half R) {
    auto h = [](float x) { return __float2half_rn(fminf(fmaxf(x, -60000.0f), 60000.0f)); };
    return fref_pack(h(A), h(Jr), h(Jz), R);
}

// 16-bit storage, staged (even nz): a block of NT threads covers the columns [z0, z0 + 2 NT)
// of RPT rows.  For each row it needs one run of columns [a, b) = [z0 - 1, z0 + 2 NT + 1)
// (clipped to the row) of the source row of every population plane, the porosity of its
// own columns and the reference words of three rows.  Thread 0 copies each run into shared
// memory with a 1-D bulk copy (cp.async.bulk) of the 16-byte-aligned window around it
// (the window may take a few elements of the neighbouring row, never of another plane:
// planes are multiples of 64 elements), completion counted in bytes on an mbarrier per
// buffer; the next row's copies are in flight while the current row computes from the
// other buffer.  Reference words live in a ring of four rows (row mod 4; the pipe axis
// row's mirror row -1 holds row 0's words), so each row after the first copies one new
// row of them.  At a closed z end the clipped runs serve every stored lane (a lane on an
// end column is not stored, as in update_pair; it reads one column past the run, inside
// the shared block, and computes on whatever it finds there);
// blocks at a periodic z end run update_pair.  Every wait is bounded: a wait that runs
// out sets *status to LBM_ERR_TIMEOUT, and the block then waits (with the drain bound)
// for the copies it has in flight and stops.
constexpr int STAGE_SPIN = 1 << 22;   // try_wait rounds of one bounded wait (a few seconds)
template <int NT>
struct __align__(16) PairStage {
    static constexpr int F = 2 * NT + 16, G = 2 * NT + 8, Q = 2 * NT + 4, P = 2 * NT + 4;   // window capacities
    uint4 pad;                   // column -1 of the first window (read by an unstored lane) lands here
    unsigned short f[2][9][F];   // 16-bit flow sources, two rows in flight
    float g[2][5][G];            // thermal sources
    float ph[2][P];              // porosity of the own columns
    uint2 q[4][Q];               // reference words, ring over row mod 4
    unsigned long long bar[2];   // one mbarrier per buffer
};

// The 16-byte-aligned window of elements (U per 16 bytes, ES bytes each) around columns
// [a, b) of row R of a plane with row stride nz: its first element, the window index of
// column a, and its length in bytes.
struct Win {
    int start, off;
    uint32_t bytes;
};
template <int U, int ES>
__device__ __forceinline__ Win win(int R, int nz, int a, int b) {
    const int e0 = R * nz + a, s = e0 & -U, e1 = (R * nz + b + U - 1) & -U;
    return {s, e0 - s, (uint32_t)((e1 - s) * ES)};
}

__device__ __forceinline__ uint32_t sm_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     sm_addr(dst)),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
// Bounded wait for the completion of phase `phase` of an mbarrier.
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t phase, int spin) {
    for (int i = 0; i < spin; ++i) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(phase)
            : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ V2 h16x2(uint32_t w, const __half*) {
    return {__half22float2(*reinterpret_cast<const __half2*>(&w))};
}
__device__ __forceinline__ V2 h16x2(uint32_t w, const __nv_bfloat16*) {
    return {__bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w))};
}
__device__ __forceinline__ float h16(unsigned short u, const __half*) { return __half2float(__ushort_as_half(u)); }
__device__ __forceinline__ float h16(unsigned short u, const __nv_bfloat16*) {
    return __bfloat162float(__ushort_as_bfloat16(u));
}
__device__ __forceinline__ Q2 q2_of(uint2 ua, uint2 ub) {
    const Qf x = fref_unpack(ua), y = fref_unpack(ub);
    return {v2(x.A, y.A), v2(x.Jr, y.Jr), v2(x.Jz, y.Jz), v2(x.R, y.R)};
}

// One staged block: rows r0 .. r0 + RPT - 1 (at most), columns z0 .. z0 + 2 NT - 1 (see above).
// spin: try_wait rounds of the per-row waits (the final drain always uses STAGE_SPIN).
// ALN: nz is a multiple of 8 and the blocks at both z ends run update_pair, so every staged
// block starts its runs at column z0 - 1 = 7 mod 8 of a row that starts 16-byte aligned
// (the window index of each column is a constant offset from it) and stores both lanes of
// every thread.
template <int STO, int NT, bool ALN>
__device__ __forceinline__ void stage_block(const Consts<float>& c, const Buf<STO>& A, const Buf<STO>& B,
                                            const float* __restrict__ phi, int plane, int r0, int RPT, int z0,
                                            int spin, int* __restrict__ status, PairStage<NT>& sb) {
    using TF = typename St<STO>::TF;
    const int nz = c.nz, t = threadIdx.x, kz0 = z0 + 2 * t;
    if (nz & 1) {   // launched for even nz only: the pair reads below assume it
        if (t == 0) atomicExch(status, LBM_ERR_INVALID);
        return;
    }
    if ((ALN && (z0 == 0 || z0 + 2 * NT + 8 > nz)) || (c.periodic && (z0 == 0 || z0 + 2 * NT >= nz))) {   // global loads
        if (kz0 < nz) update_pair<STO, true>(c, A, B, phi, plane, r0, RPT, kz0);
        return;
    }
    const bool row0_wall = c.geometry == ANNULUS || c.geometry == ANNULUS_PERIODIC_Z;
    const auto computes = [&](int kr) { return kr < c.nr - 1 && (kr > 0 || !row0_wall); };
    const TF* __restrict__ F = A.f;
    const float* __restrict__ G = A.g;
    const uint2* __restrict__ Qp = c.fref;
    const int rows = min(RPT, c.nr - r0);
    const int a = ALN ? z0 - 1 : max(z0 - 1, 0);   // first column of the runs; they end at min(z0 + 2 NT + 1, nz)
    const uint32_t bar0 = sm_addr(&sb.bar[0]), bar1 = sm_addr(&sb.bar[1]);
    if (t == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar0) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar1) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    // thread 0: copy the sources of row r0 + j into buffer j & 1, and the reference words
    // it needs first (rows kr - 1 .. kr + 1 for the first row, then row kr + 1)
    const auto issue = [&](int j) {
        const int kr = r0 + j, bf = j & 1;
        const uint32_t bar = bf ? bar1 : bar0;
        const int q_lo = j == 0 ? kr - 1 : kr + 1, q_hi = min(kr + 1, c.nr - 1);
        const bool axis = kr == 0 && !row0_wall;   // pipe axis: row -1 mirrors row 0
        const bool comp = computes(kr);
        const int Rm = axis ? kr : kr - 1, b = min(z0 + 2 * NT + 1, nz), pb = min(z0 + 2 * NT, nz);
        const Win wf[3] = {win<8, 2>(Rm, nz, a, b), win<8, 2>(kr, nz, a, b), win<8, 2>(kr + 1, nz, a, b)};
        const Win wg[3] = {win<4, 4>(Rm, nz, a, b), win<4, 4>(kr, nz, a, b), win<4, 4>(kr + 1, nz, a, b)};
        const Win wp = win<4, 4>(kr, nz, z0, pb);
        uint32_t bytes = 0;
        if (comp)   // three flow slots per row group; thermal slots 0, 2, 4 in row kr, 1 and 3 in the others
            bytes = 3 * (wf[0].bytes + wf[1].bytes + wf[2].bytes) + 3 * wg[1].bytes + wg[0].bytes + wg[2].bytes +
                    wp.bytes;
        for (int qr = q_lo; qr <= q_hi; ++qr)
            if (qr >= 0 || axis) bytes += win<2, 8>(max(qr, 0), nz, a, b).bytes;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // after the reads of the buffer's last use
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
        if (comp) {
            const int p1 = axis ? 3 : 1, p5 = axis ? 6 : 5, p8 = axis ? 7 : 8;
            // flow slot i: plane and row group (0: row kr - 1 or its mirror, 1: kr, 2: kr + 1)
            const int fpl[9] = {0, p1, 2, 3, 4, p5, 6, 7, p8};
            const int frg[9] = {1, 0, 1, 2, 1, 0, 2, 2, 0};
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const Win& w = wf[frg[i]];
                bulk_copy(sb.f[bf][i], F + fpl[i] * plane + w.start, w.bytes, bar);
            }
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                const Win& w = wg[frg[i]];
                bulk_copy(sb.g[bf][i], G + fpl[i] * plane + w.start, w.bytes, bar);
            }
            bulk_copy(sb.ph[bf], phi + wp.start, wp.bytes, bar);
        }
        for (int qr = q_lo; qr <= q_hi; ++qr)
            if (qr >= 0 || axis) {
                const Win w = win<2, 8>(max(qr, 0), nz, a, b);
                bulk_copy(sb.q[qr & 3], Qp + w.start, w.bytes, bar);
            }
    };
    if (t == 0) issue(0);
    const bool active = ALN || kz0 < nz;
    bool ok = true;
#pragma unroll 1
    for (int j = 0; j < rows; ++j) {
        if (t == 0 && j + 1 < rows) issue(j + 1);
        const int kr = r0 + j, bf = j & 1;
        ok = bar_wait(bf ? bar1 : bar0, (j >> 1) & 1, spin);
        if (active && computes(kr)) {
            const bool axis = kr == 0;
            const int p1 = axis ? 3 : 1, p5 = axis ? 6 : 5, p8 = axis ? 7 : 8;
            const int Rm = axis ? kr : kr - 1;
            // window index of the own column kz0 in row group rg (the left column is one
            // below, the right columns one and two above)
            const auto wo = [&](int R, int U) { return kz0 - a + (ALN ? U - 1 : ((R * nz + a) & (U - 1))); };
            const int of[3] = {wo(Rm, 8), wo(kr, 8), wo(kr + 1, 8)};
            const int og[3] = {wo(Rm, 4), wo(kr, 4), wo(kr + 1, 4)};
            const auto own = [&](int i, int rg) {
                return h16x2(*reinterpret_cast<const uint32_t*>(&sb.f[bf][i][of[rg]]), F);
            };
            const auto fat = [&](int i, int rg, int d) {   // columns kz0 + d, kz0 + d + 1
                return v2(h16(sb.f[bf][i][of[rg] + d], F), h16(sb.f[bf][i][of[rg] + d + 1], F));
            };
            const auto gown = [&](int i, int rg) { return V2{*reinterpret_cast<const float2*>(&sb.g[bf][i][og[rg]])}; };
            const auto gat = [&](int i, int rg, int d) {
                return v2(sb.g[bf][i][og[rg] + d], sb.g[bf][i][og[rg] + d + 1]);
            };
            V2 fh[9], gh[5];
            fh[0] = own(0, 1);
            fh[1] = own(1, 0);
            fh[2] = fat(2, 1, -1);
            fh[3] = own(3, 2);
            fh[4] = fat(4, 1, 1);
            fh[5] = fat(5, 0, -1);
            fh[6] = fat(6, 2, -1);
            fh[7] = fat(7, 2, 1);
            fh[8] = fat(8, 0, 1);
            gh[0] = gown(0, 1);
            gh[1] = gown(1, 0);
            gh[2] = gat(2, 1, -1);
            gh[3] = gown(3, 2);
            gh[4] = gat(4, 1, 1);
            const V2 ph{*reinterpret_cast<const float2*>(&sb.ph[bf][kz0 - z0 + (ALN ? 0 : (kr * nz + z0) & 3)])};
            const auto qw = [&](int rs, int cs) {
                const int qr = kr - 1 + rs;
                const uint2* q = sb.q[qr & 3];
                const int o = kz0 - a + (ALN ? 1 : ((max(qr, 0) * nz + a) & 1));
                const uint4 u = *reinterpret_cast<const uint4*>(q + o);   // the own pair's two words
                if (cs == 1) return q2_of(make_uint2(u.x, u.y), make_uint2(u.z, u.w));
                if (cs == 0) return q2_of(q[o - 1], make_uint2(u.x, u.y));
                return q2_of(make_uint2(u.z, u.w), q[o + 2]);
            };
            const bool st0 = ALN || kz0 > 0 || c.periodic, st1 = ALN || kz0 + 1 < nz - 1 || c.periodic;
            pair_finish<STO, true>(c, B, plane, kr, kr * nz, kz0, p1, p5, p8, fh, gh, ph, qw, st0, st1);
        }
        if (__syncthreads_or(!ok)) {   // a wait ran out: drain what is in flight and stop
            if (t == 0) {
                atomicExch(status, LBM_ERR_TIMEOUT);
                bar_wait(bf ? bar1 : bar0, (j >> 1) & 1, STAGE_SPIN);
                if (j + 1 < rows) bar_wait(bf ? bar0 : bar1, ((j + 1) >> 1) & 1, STAGE_SPIN);
            }
            return;
        }
    }
}
