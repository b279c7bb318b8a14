// lbm_two.cuh -- two time steps per pass over the state, FP32 storage.
//
// One step reads and writes every population once (118 bytes per node) and does about 330
// operations on them: it is bound by memory on large grids and by its launches on small ones.
// Here the state between the two steps never leaves the SM: a warp takes a strip of 64 columns
// (two z-adjacent nodes per thread) and marches over rows.  At row j it updates the strip's row j
// from the state in memory (first step) and then row j - 1 (second step), whose sources are
// rows j - 2 .. j of the first step:
//   e_r = +1 populations of row j - 2, e_r = 0 populations of row j - 1 (both kept in shared
//   memory, a slot per thread) and e_r = -1 populations of row j (registers).
// Columns are exchanged inside the warp: every thread loads its own two columns of a source
// plane as one vector load, and the e_z = +-1 populations move one column by a shuffle.
// The outermost column is wrong after the first step and the next one after the second, so
// a strip stores its inner 60 columns; strips overlap by four.  No barrier, no wait.
//
// Boundary nodes are part of the pass (the one-step path has its own kernel for them): a
// boundary node's update needs the pulled state of its interior neighbour (Sec. 4, ref.
// [47]), which is the same row's neighbouring column (end columns: the other lane of the
// pair, or with odd nz the previous thread) or the neighbouring row (wall rows: the row that
// is pulled is the neighbour's).  Wall rows of the second step are marches of their own over
// the one neighbouring row, so that the main march carries no extra state.
//
// 16-bit storage takes single steps: its results hang on the rounding of every stored value,
// and a pass evaluated in another order of operations decorrelates those roundings within a
// few steps (measured after 20 steps with BF16: 1e-4 relative in u between the two orders, the
// size of the format's own error), while the time it won was 12 % (0.41 against 0.46 ms per
// step, 4096 x 8192, FP16).
#pragma once
#include "lbm_f32.h"
#include "lbm_pair.cuh"

namespace lbm {

// Row constants (RowC) and c_s^2 2 (tau - 1/2) / r^2.
struct Row32 : RowC {
    float c2rr;
};
__device__ __forceinline__ Row32 row_consts32(const Consts32& c, int kr) {
    Row32 q;
    static_cast<RowC&>(q) = row_consts(c, kr);
    q.c2rr = q.c2r * q.inv_r;
    return q;
}

constexpr int TWO_THREADS = 128;
constexpr int TWO_COLS = 60;   // columns a strip stores (64 loaded)
constexpr int TWO_KEEP = 17;   // 16-byte slots (two pairs) a thread keeps from row to row
constexpr unsigned FULL = 0xffffffffu;

// A factor or addend that both lanes share: two scalar instructions, which take it from the
// constant bank, as an immediate or from one register, where the packed form first needs it in
// a register pair; they cost the FMA pipe the same two cycles.  (The kernels of 16-bit storage
// keep the packed form: their results hang on it bit by bit, and it needs fewer registers there.)
struct Both { float v; };
__device__ __forceinline__ Both both(float v) { return {v}; }
__device__ __forceinline__ V2 operator+(V2 a, Both b) { return v2(__fadd_rn(a.v.x, b.v), __fadd_rn(a.v.y, b.v)); }
__device__ __forceinline__ V2 operator*(V2 a, Both b) { return v2(__fmul_rn(a.v.x, b.v), __fmul_rn(a.v.y, b.v)); }
__device__ __forceinline__ V2 fma2(V2 a, Both b, V2 c) {
    return v2(__fmaf_rn(a.v.x, b.v, c.v.x), __fmaf_rn(a.v.y, b.v, c.v.y));
}
__device__ __forceinline__ V2 fma2(V2 a, V2 b, Both c) {
    return v2(__fmaf_rn(a.v.x, b.v.x, c.v), __fmaf_rn(a.v.y, b.v.y, c.v));
}
__device__ __forceinline__ V2 fma2(V2 a, Both b, Both c) {
    return v2(__fmaf_rn(a.v.x, b.v, c.v), __fmaf_rn(a.v.y, b.v, c.v));
}
// The arithmetic below is written once for a pair (V = V2) and for a single node (V = float).
__device__ __forceinline__ float operator+(float a, Both b) { return __fadd_rn(a, b.v); }
__device__ __forceinline__ float operator*(float a, Both b) { return __fmul_rn(a, b.v); }
__device__ __forceinline__ float fma2(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float fma2(float a, Both b, float c) { return __fmaf_rn(a, b.v, c); }
__device__ __forceinline__ float fma2(float a, float b, Both c) { return __fmaf_rn(a, b, c.v); }
__device__ __forceinline__ float fma2(float a, Both b, Both c) { return __fmaf_rn(a, b.v, c.v); }
__device__ __forceinline__ V2 rcp_few(V2 x) { return rcp_fast(x); }       // reciprocal, square root: hardware
__device__ __forceinline__ float rcp_few(float x) { return rcp_approx(x); }   // approximations
__device__ __forceinline__ V2 sqrt_few(V2 x) { return sqrt_fast(x); }
__device__ __forceinline__ float sqrt_few(float x) { return sqrt_approx(x); }
template <class V> __device__ __forceinline__ V rcp_newton(V x) {   // and one Newton step (rcp_acc)
    const V y = rcp_few(x);
    return fma2(y, fma2(-x, y, both(1.0f)), y);
}
template <class V> __device__ __forceinline__ V all(float x);
template <> __device__ __forceinline__ V2 all<V2>(float x) { return v2(x); }
template <> __device__ __forceinline__ float all<float>(float x) { return x; }

// Sums and differences of a pair's populations, shared by the recovery and the collision
// (both are written on them; a packed multiply-add takes two issue cycles of the FMA pipe, the
// pipe that bounds this code, so operations are what is saved: about 175 per pair and step
// against 265 with the moments of Eq. 18 formed one by one).
template <class V> struct Sums {
    V a, b;         // f_1 + .. + f_4, f_5 + .. + f_8
    V s7, s8;       // m_7 = (f_1 + f_3) - (f_2 + f_4), m_8 = (f_5 + f_7) - (f_6 + f_8)
    V d13, d24;     // f_1 - f_3, f_2 - f_4
    V jr, jz;       // m_3, m_5
    V m0;
};

template <class V> __device__ __forceinline__ Sums<V> sums2(const V* fh) {
    Sums<V> s;
    const V s13 = fh[1] + fh[3], s24 = fh[2] + fh[4], s57 = fh[5] + fh[7], s68 = fh[6] + fh[8];
    const V x57 = fh[5] - fh[7], x68 = fh[6] - fh[8];
    s.a = s13 + s24;
    s.b = s57 + s68;
    s.s7 = s13 - s24;
    s.s8 = s57 - s68;
    s.d13 = fh[1] - fh[3];
    s.d24 = fh[2] - fh[4];
    s.jr = s.d13 + (x57 - x68);
    s.jz = s.d24 + (x57 + x68);
    s.m0 = fh[0] + (s.a + s.b);
    return s;
}

// Eq. 8 per node (porous() of lbm_physics.cuh) for two nodes.
template <class V>
__device__ __forceinline__ void porous_two(const Consts32& c, V phi, V& lin, V& nl, V& inv_phi) {
    const V ph2 = phi * phi;
    const V ip3 = rcp_few(ph2 * phi);
    inv_phi = ph2 * ip3;
    if (c.porous_mode == 2) {
        const V om = fma2(phi, both(-1.0f), both(1.0f));
        lin = (om * om) * both(c.lin_coef) * ip3;
        nl = c.ergun ? om * both(c.nl_coef) * ip3 : om * both(c.nl_coef) * sqrt_few(ip3);
    } else if (c.porous_mode == 1) {
        lin = all<V>(c.lin_coef);
        nl = c.ergun ? sqrt_few(ip3) * both(c.nl_coef) : all<V>(c.nl_coef);
    } else {
        lin = all<V>(0.f);
        nl = all<V>(0.f);
    }
}

// recover() of lbm_physics.cuh (Eq. 26-30, 38) for two nodes; dT is relative to each
// node's reference temperature T0 + R(x), rref = R(x).
template <class V>
__device__ __forceinline__ void recover_two(const Consts32& c, const Row32& q, V phi, V lin, V nl,
                                            const Sums<V>& s, const V* gh, V rref, V& rho, V& ur, V& uz, V& dT) {
    dT = ((gh[0] + gh[1]) + (gh[2] + gh[3])) + gh[4];
    rho = fma2(s.m0, both(q.inv_r), both(1.0f));
    const V Gz = fma2(dT + rref, both(c.gbeta), both(c.az));
    const V inv_rho = rcp_newton(rho);
    const V vr = fma2(s.m0, both(q.c1), s.jr) * inv_rho;
    const V hp = phi * both(q.hr);
    const V vz = fma2(s.jz, inv_rho, hp * Gz);
    const V hd = phi * both(q.qr) * lin;
    const V lr0 = hd + both(q.L0r);
    const V lz0 = hd + both(q.hr);
    // Eq. 28 as in recover(), without a branch: x = 0 (no Forchheimer drag) adds 0
    const V x = hp * nl * sqrt_few(fma2(vr, vr, vz * vz));
    const V Dr = fma2(x, rcp_few(lr0 + sqrt_few(fma2(lr0, lr0, x))), lr0 + lr0);
    const V Dz = fma2(x, rcp_few(lz0 + sqrt_few(fma2(lz0, lz0, x))), lz0 + lz0);
    ur = vr * rcp_newton(Dr);
    uz = vz * rcp_newton(Dz);
}

// collide() of lbm_physics.cuh (Eq. 6, 21-25, 33-37) for two nodes, in place; rref = R(x).
// The change dm = m+ - m of Eq. 21 in the combinations M^-1 needs, with S of Eq. 24 and m_eq of
// Eq. 19-20 put in: with P = u_r F~_r, Q = u_z F~_z, R = r rho / phi and s_e = s_eps,
//   dm_1 / 36 = -(s_e / 36) (-2 f_0 + a + 4 b) + G,  dm_2 / 36 = -(s_e / 12) (f_0 - a) - G,
//   G = R (s_e u^2 / 12 + h_e (P + Q) / 6),
//   dm_7 / 4 = -(s_nu / 4) m_7 + R (s_nu (u_r^2 - u_z^2) / 4 + h_nu (P - Q) / 2),
//   dm_8 / 4 = -(s_nu / 4) m_8 + R (s_nu u_r u_z / 4 + h_nu (u_r F~_z + u_z F~_r) / 4),
//   m_4 = m_3 - 3 (f_1 - f_3), m_6 = m_5 - 3 (f_2 - f_4).
// As in collide(), Eq. 22 is applied to the change only, and mass and momentum of the change
// are sums of exact multiples of its four parts.
template <class V>
__device__ __forceinline__ void collide_two(const Consts32& c, const Row32& q, V phi, V lin, V nl, V inv_phi,
                                            const Sums<V>& s, V* fh, V* gh, V rref, V rho, V ur, V uz, V dT) {
    const V Tb = rref + both(c.T0);   // the nodes' reference temperatures
    const V T = Tb + dT;
    const V uz2 = uz * uz;
    const V u2 = fma2(ur, ur, uz2), ud = fma2(ur, ur, -uz2);
    const V Gz = fma2(dT + rref, both(c.gbeta), both(c.az));
    const V pd = phi * fma2(nl, sqrt_few(u2), lin);
    const V kr = pd + both(q.c2rr);
    const V Ftr = fma2(-kr, ur, both(q.cs2r));   // Eq. 25
    const V Ftz = fma2(-pd, uz, phi * Gz);
    const V rr = rho * both(q.r);
    const V rri = rr * inv_phi;
    const V e3 = rr * ur, e5 = rr * uz;
    // S_3 without its rest constant c_s^2 (see collide()), S_5
    const V S3 = fma2(-kr, e3, s.m0 * both(q.cs2r));
    const V S5 = rr * Ftz;
    const V uzFz = uz * Ftz;
    const V pq = fma2(ur, Ftr, uzFz), pm = fma2(ur, Ftr, -uzFz);
    const V G = rri * fma2(u2, both(c.g_u), pq * both(c.g_f));
    const V A1 = fma2(fma2(fh[0], both(-2.0f), fma2(s.b, both(4.0f), s.a)), both(-c.a_e), G);
    const V A2 = fma2(fh[0] - s.a, both(-c.g_u), -G);
    const V b14 = fma2(A2, both(-2.0f), -A1), b58 = fma2(A1, both(2.0f), A2);
    const V a7 = fma2(s.s7, both(-c.a_nu), rri * fma2(ud, both(c.a_nu), pm * both(c.b7)));
    const V a8 = fma2(s.s8, both(-c.a_nu), rri * fma2(ur * uz, both(c.a_nu), fma2(ur, Ftz, uz * Ftr) * both(c.b8)));
    const V a3 = fma2(s.jr - e3, both(-c.a_j), S3 * both(c.b_j));
    const V a4 = fma2(fma2(s.d13, both(-3.0f), s.jr + e3), both(-c.a_q), S3 * both(-c.b_q));
    const V a5 = fma2(s.jz - e5, both(-c.a_j), S5 * both(c.b_j));
    const V a6 = fma2(fma2(s.d24, both(-3.0f), s.jz + e5), both(-c.a_q), S5 * both(-c.b_q));
    const V x3 = fma2(a4, both(-2.0f), a3), x5 = fma2(a6, both(-2.0f), a5);
    const V y3 = a3 + a4, y5 = a5 + a6;
    const V yp = y3 + y5, ym = y3 - y5;
    const V bp = b14 + a7, bm = b14 - a7, cp = b58 + a8, cm = b58 - a8;
    fh[0] = fma2(A2 - A1, both(4.0f), fh[0]);
    fh[1] += bp + x3;
    fh[2] += bm + x5;
    fh[3] += bp - x3;
    fh[4] += bm - x5;
    fh[5] += cp + yp;
    fh[6] += cm - ym;
    fh[7] += cp - yp;
    fh[8] += cm + ym;
    // D2Q5 (Eq. 33, 35-37), relative to T0 + R(x)
    const float wd = c.wg_den, wp = (1.0f + q.kT) * wd, wm = (1.0f - q.kT) * wd;
    const V cu = ur * both(-q.inv_r);
    const V hT = T * both(0.5f);
    const V Tr = hT * ur, Tz = hT * uz;
    const V t1 = dT * both(0.1f);
    const V g1e = t1 + Tr, g3e = t1 - Tr;
    const V g2e = t1 + Tz, g4e = t1 - Tz;
    const V g0e = fma2(t1, both(-4.0f), dT);
    const V wT0 = Tb * both(0.6f), wT1 = Tb * both(0.1f);
    gh[0] = fma2(cu, g0e + wT0, fma2(gh[0] - g0e, both(-wd), gh[0]));
    gh[1] = fma2(cu, g1e + wT1, fma2(gh[1] - g1e, both(-wp), gh[1]));
    gh[2] = fma2(cu, g2e + wT1, fma2(gh[2] - g2e, both(-wd), gh[2]));
    gh[3] = fma2(cu, g3e + wT1, fma2(gh[3] - g3e, both(-wm), gh[3]));
    gh[4] = fma2(cu, g4e + wT1, fma2(gh[4] - g4e, both(-wd), gh[4]));
}

// The pair one column to the left (e_z = +1: column c takes column c - 1) or right.
__device__ __forceinline__ V2 from_left(V2 x) { return v2(__shfl_up_sync(FULL, x.v.y, 1), x.v.x); }
__device__ __forceinline__ V2 from_right(V2 x) { return v2(x.v.y, __shfl_down_sync(FULL, x.v.x, 1)); }

// Boundary rebuild (rebuild_flow, rebuild_thermal of lbm_physics.cuh) of the boundary lanes
// (w0, w1; classes k0, k1) of row j from the pulled state of row p (p = j except on wall rows):
// fh, gh, m0, rho, ur, uz, dT hold that state with its reference reff and 1/phi iphf, and receive
// the boundary state on the boundary lanes.  nb(x): the interior neighbours' values, lane by
// lane.  phj, refj: porosity and temperature reference of row j.
template <class NB>
__device__ __forceinline__ void wall_rebuild(const Consts32& c, int p, int j, int k0, int k1, bool w0, bool w1,
                                             const NB& nb, V2 (&fh)[9], V2 (&gh)[5], V2 m0, V2& rho, V2& ur, V2& uz,
                                             V2& dT, V2 iphf, V2 reff, V2 phj, V2 refj) {
    const auto put = [&](V2& x, V2 w) { x = v2(w0 ? w.v.x : x.v.x, w1 ? w.v.y : x.v.y); };
    const float rf = c.r0 + float(p), rb = c.r0 + float(j);
    const float inv_rf = rcp_acc(rf), inv_rb = rcp_acc(rb);
    const V2 m0f = nb(m0), rhof = nb(rho), urf = nb(ur), uzf = nb(uz), dTf = nb(dT), Rf = nb(reff), ipf = nb(iphf);
    const V2 drho = m0f * inv_rf;
    V2 drhob = drho, rhob = rhof, urb = v2(0.f), uzb = v2(0.f);
    const bool pipe = c.geometry == PIPE_INFLOW;
    V2 ipb = v2(1.0f);
    if (pipe) {   // inlet: u = (0, u_in); outlet: u of the neighbour, density 1; their own 1/phi
        ipb = rcp_acc(phj);
        const bool o0 = k0 == OUTLET, o1 = k1 == OUTLET;
        urb = v2(o0 ? urf.v.x : 0.f, o1 ? urf.v.y : 0.f);
        uzb = v2(o0 ? uzf.v.x : (k0 == INLET ? c.u_in : 0.f), o1 ? uzf.v.y : (k1 == INLET ? c.u_in : 0.f));
        drhob = v2(o0 ? 0.f : drho.v.x, o1 ? 0.f : drho.v.y);
        rhob = v2(o0 ? 1.f : rhof.v.x, o1 ? 1.f : rhof.v.y);
    }
    const V2 u2f = (1.5f * fma2(urf, urf, uzf * uzf)) * ipf, u2b = (1.5f * fma2(urb, urb, uzb * uzb)) * ipb;
    V2 mb = v2(0.f);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const auto e_dot = [&](V2 r, V2 z) {
            V2 e = v2(0.f);
            if (ex9(i) == 1) e = r;
            if (ex9(i) == -1) e = -r;
            if (ez9(i) == 1) e = ex9(i) ? e + z : z;
            if (ez9(i) == -1) e = ex9(i) ? e - z : -z;
            return e;
        };
        const V2 eu = e_dot(urf, uzf);
        const V2 q = fma2(rhof, fma2(eu, fma2(4.5f * ipf, eu, v2(3.0f)), -u2f), drho);
        V2 qb = drhob;
        if (pipe) {
            const V2 eb = e_dot(urb, uzb);
            qb = fma2(rhob, fma2(eb, fma2(4.5f * ipb, eb, v2(3.0f)), -u2b), drhob);
        }
        const V2 w = fma2(rb * w9<float>(i), qb, nb(fh[i])) - (rf * w9<float>(i)) * q;
        mb += w;
        put(fh[i], w);
    }
    const float Th = c.T_hot - c.T0, Tc = c.T_cold - c.T0;
    const auto wall_T = [&](int k, float d, float rfb, float own) {
        return (k == WALL_IN || k == INLET) ? Th - own : k == WALL_OUT ? Tc - own : (d + rfb) - own;
    };
    const V2 dTb = v2(wall_T(k0, dTf.v.x, Rf.v.x, refj.v.x), wall_T(k1, dTf.v.y, Rf.v.y, refj.v.y));
    const V2 hTf = 0.5f * (c.T0 + Rf + dTf), hTb = 0.5f * (c.T0 + refj + dTb);
    const V2 tr = hTb * urb - hTf * urf, tz = hTb * uzb - hTf * uzf;
    const V2 d = dTb - dTf;
    const V2 t1 = 0.1f * d;
    const V2 g[5] = {nb(gh[0]) + fma2(t1, -4.0f, d), nb(gh[1]) + (t1 + tr), nb(gh[2]) + (t1 + tz),
                     nb(gh[3]) + (t1 - tr), nb(gh[4]) + (t1 - tz)};
#pragma unroll
    for (int i = 0; i < 5; ++i) put(gh[i], g[i]);
    put(rho, fma2(mb, inv_rb, v2(1.0f)));
    put(ur, urb);
    put(uz, uzb);
    put(dT, dTb);
}

// The same where the neighbour of an end column sits in the other lane of the pair or (ODD: odd
// nz) in the previous thread; ca: the pair's first column.
template <bool ODD>
__device__ __forceinline__ void wall_pair(const Consts32& c, int p, int j, int ca, V2 (&fh)[9], V2 (&gh)[5],
                                          V2 m0, V2& rho, V2& ur, V2& uz, V2& dT, V2 iphf, V2 reff, V2 phj, V2 refj) {
    const int nz = c.nz, cb = ca + 1;
    const bool closed = !c.periodic;
    const int k0 = node_class(c.geometry, c.nr, nz, j, ca), k1 = node_class(c.geometry, c.nr, nz, j, cb);
    // (periodic z: only wall rows come here, and the columns past the ends are wrapped ones)
    const bool w0 = (!closed || (ca >= 0 && ca < nz)) && is_wall(k0);
    const bool w1 = (!closed || (cb >= 0 && cb < nz)) && is_wall(k1);
    const bool l_first = closed && ca == 0, h_last = closed && cb == nz - 1;
    const bool l_last = ODD && closed && ca == nz - 1;
    const auto nb = [&](V2 x) {
        float up = 0.f;
        if (ODD) up = __shfl_up_sync(FULL, x.v.y, 1);
        return v2(l_first ? x.v.y : (l_last ? up : x.v.x), h_last ? x.v.x : x.v.y);
    };
    wall_rebuild(c, p, j, k0, k1, w0, w1, nb, fh, gh, m0, rho, ur, uz, dT, iphf, reff, phj, refj);
}

// Two columns of a plane (VEC: aligned neighbours), and the stores of both or the first.
template <bool VEC> __device__ __forceinline__ V2 ld_two(const float* p, int la, int lb) {
    if (VEC) return {*reinterpret_cast<const float2*>(p + la)};
    return v2(p[la], p[lb]);
}
template <bool VEC> __device__ __forceinline__ void st_two(float* p, V2 v, bool second) {
    if (VEC) {
        *reinterpret_cast<float2*>(p) = v.v;
    } else {
        p[0] = v.v.x;
        if (second) p[1] = v.v.y;
    }
}
// Two columns of the reference plane R(x), as loaded and as floats.
template <bool VEC> __device__ __forceinline__ uint32_t ld_ref(const __half* p, int la, int lb) {
    if (VEC) return *reinterpret_cast<const uint32_t*>(p + la);
    const auto* q = reinterpret_cast<const unsigned short*>(p);
    return (uint32_t)q[la] | ((uint32_t)q[lb] << 16);
}
__device__ __forceinline__ V2 ref_of(uint32_t w) { return {__half22float2(*reinterpret_cast<const __half2*>(&w))}; }

// March of one warp: rows ka .. kb of the state two steps on, columns s TWO_COLS ..
// (s + 1) TWO_COLS - 1 (an end column that would be alone in a strip of its own belongs to the
// strip before: two_plan); wall >= 0: ka = kb is the neighbour row of wall row `wall`, and that wall
// row is written instead.  VEC: nz even.  WALLS: the march meets boundary nodes.
template <bool VEC, bool WALLS>
__device__ __forceinline__ void two_march(const Consts32& c, const State32& A, const State32& B,
                                          const float* __restrict__ phi, int plane, int s, int ka, int kb, int wall,
                                          float4* __restrict__ ring) {
    const int nr = c.nr, nz = c.nz, lane = threadIdx.x & 31;
    const int c0 = s * TWO_COLS - 2, ca = c0 + 2 * lane;
    const bool closed = !c.periodic;
    // columns loaded: wrapped when periodic, clamped into the row otherwise (such lanes are
    // only read by lanes that are not stored)
    int la, lb;
    if (closed) {
        la = VEC ? min(max(ca, 0), nz - 2) : min(max(ca, 0), nz - 1);
        lb = VEC ? la + 1 : min(max(ca + 1, 0), nz - 1);
    } else {
        la = (ca + nz) % nz;
        lb = VEC ? la + 1 : (ca + 1 + nz) % nz;
    }
    const bool edge = WALLS && closed && (c0 <= 0 || c0 + 63 >= nz - 1);   // the strip holds an end column
    const bool own = lane >= 1 && (lane <= 30 || (!VEC && closed && ca == nz - 1));
    const bool st0 = own && ca < nz, st1 = own && ca + 1 < nz;
    const bool row0_wall = c.geometry == ANNULUS || c.geometry == ANNULUS_PERIODIC_Z;
    const float* __restrict__ F = A.f;
    const float* __restrict__ G = A.g;
    // what the second step of a row takes from earlier rows, in shared memory, one slot per
    // thread each (no exchange between threads): e_r = 0 populations of the last row (f_0, f_2,
    // f_4, g_0, g_2, g_4), e_r = +1 populations (f_1, f_5, f_8, g_1) of the last two rows, row j
    // in the half of its parity, and a row's re-referencing terms, porosity coefficients and
    // reference (row j again in the half of its parity)
    float4* const keep = ring + threadIdx.x;
    const auto put = [&](int slot, V2 a, V2 b) {
        keep[slot * TWO_THREADS] = make_float4(a.v.x, a.v.y, b.v.x, b.v.y);
    };
    const auto take = [&](int slot, V2& a, V2& b) {
        const float4 t = keep[slot * TWO_THREADS];
        a = v2(t.x, t.y);
        b = v2(t.z, t.w);
    };
    const auto swap = [&](int slot, V2& oa, V2& ob, V2 a, V2 b) {
        take(slot, oa, ob);
        put(slot, a, b);
    };
    // the row that first-step row j pulls
    const auto pulled = [&](int j) { return !WALLS ? j : (j == nr - 1 ? nr - 2 : (j == 0 && row0_wall ? 1 : j)); };
    // The next row's sources are asked into L2 while this row computes: lanes 2 i and 2 i + 1
    // take the two 128-byte lines of plane i's source row (flow, temperature, porosity,
    // reference).
    const char* ahead;
    int ahead_row, ahead_size = 4;
    {
        const int pl = lane >> 1, i = pl < 9 ? pl : pl - 9, col = min(max(c0 + 32 * (lane & 1), 0), nz - 1);
        ahead_row = pl > 13 ? 1 : -ex9(i);
        if (pl < 9) ahead = (const char*)(F + (int64_t)i * plane + col);
        else if (pl < 14) ahead = (const char*)(G + (int64_t)i * plane + col);
        else if (pl == 14) ahead = (const char*)(phi + col);
        else ahead = (const char*)(c.tref + col), ahead_size = 2;
    }
    const auto prefetch = [&](int j) {
        const int r = min(max(j + ahead_row, 0), nr - 1);
        asm volatile("prefetch.global.L2 [%0];" ::"l"(ahead + (int64_t)r * nz * ahead_size));
    };
#pragma unroll 1
    for (int j = max(ka - 1, 0); j <= kb + 1; ++j) {
        V2 fh[9], gh[5];
        {   // first step, row j
            const int p = pulled(j);
            const bool axis = WALLS && p == 0;   // pipe axis: the e_r = +1 sources are row 0's mirror image
            const int row = p * nz, rowp = row + nz, rowm = axis ? row : row - nz;
            const int i1 = axis ? 3 : 1, i5 = axis ? 6 : 5, i8 = axis ? 7 : 8;
            const auto ld = [&](const float* q) { return ld_two<VEC>(q, la, lb); };
            fh[0] = ld(F + row);
            fh[1] = ld(F + (i1 * plane + rowm));
            fh[2] = ld(F + (2 * plane + row));
            fh[3] = ld(F + (3 * plane + rowp));
            fh[4] = ld(F + (4 * plane + row));
            fh[5] = ld(F + (i5 * plane + rowm));
            fh[6] = ld(F + (6 * plane + rowp));
            fh[7] = ld(F + (7 * plane + rowp));
            fh[8] = ld(F + (i8 * plane + rowm));
            gh[0] = ld(G + row);
            gh[1] = ld(G + (i1 * plane + rowm));
            gh[2] = ld(G + (2 * plane + row));
            gh[3] = ld(G + (3 * plane + rowp));
            gh[4] = ld(G + (4 * plane + row));
            V2 ph = ld(phi + row);
            const uint32_t wm = ld_ref<VEC>(c.tref + rowm, la, lb), wo = ld_ref<VEC>(c.tref + row, la, lb);
            const uint32_t wp = ld_ref<VEC>(c.tref + rowp, la, lb);
            if (j <= kb) prefetch(j + 1);
            V2 R = ref_of(wo), lin, nl, iph;
            porous_two(c, ph, lin, nl, iph);
            const V2 t1 = (ref_of(wm) - R) * both(0.1f), t3 = (ref_of(wp) - R) * both(0.1f);
            const V2 t2 = (from_left(R) - R) * both(0.1f), t4 = (from_right(R) - R) * both(0.1f);
            const int u = 7 + 5 * (j & 1);
            put(u, t1, t2);
            put(u + 1, t3, t4);
            put(u + 2, ph, lin);
            put(u + 3, nl, iph);
            reinterpret_cast<uint32_t&>(keep[(u + 4) * TWO_THREADS]) = wo;
            gh[1] += t1;
            gh[3] += t3;
            fh[2] = from_left(fh[2]);
            fh[5] = from_left(fh[5]);
            fh[6] = from_left(fh[6]);
            fh[4] = from_right(fh[4]);
            fh[7] = from_right(fh[7]);
            fh[8] = from_right(fh[8]);
            gh[2] = from_left(gh[2]) + t2;
            gh[4] = from_right(gh[4]) + t4;
            V2 rho, ur, uz, dT;
            Sums<V2> sm = sums2(fh);
            recover_two(c, row_consts32(c, p), ph, lin, nl, sm, gh, R, rho, ur, uz, dT);
            if (WALLS && (edge || p != j)) {
                const V2 Rf = R, iphf = iph;
                if (p != j) {
                    ph = ld_two<VEC>(phi + j * nz, la, lb);
                    R = ref_of(ld_ref<VEC>(c.tref + j * nz, la, lb));
                    porous_two(c, ph, lin, nl, iph);
                }
                wall_pair<!VEC>(c, p, j, ca, fh, gh, sm.m0, rho, ur, uz, dT, iphf, Rf, ph, R);
                sm = sums2(fh);
            }
            collide_two(c, row_consts32(c, j), ph, lin, nl, iph, sm, fh, gh, R, rho, ur, uz, dT);
            fh[2] = from_left(fh[2]);
            fh[5] = from_left(fh[5]);
            fh[6] = from_left(fh[6]);
            gh[2] = from_left(gh[2]);
            fh[4] = from_right(fh[4]);
            fh[7] = from_right(fh[7]);
            fh[8] = from_right(fh[8]);
            gh[4] = from_right(gh[4]);
        }
        const int par = 3 + 2 * (j & 1);
        V2 f[9], g[5];
        f[3] = fh[3];
        f[6] = fh[6];
        f[7] = fh[7];
        g[3] = gh[3];
        swap(0, f[0], f[2], fh[0], fh[2]);
        swap(1, f[4], g[0], fh[4], gh[0]);
        swap(2, g[2], g[4], gh[2], gh[4]);
        swap(par, f[1], f[5], fh[1], fh[5]);
        swap(par + 1, f[8], g[1], fh[8], gh[1]);
        if (WALLS && j == 0 && !row0_wall) {   // pipe axis: row -1 is the mirror image of row 0
            put(5, fh[3], fh[6]);
            put(6, fh[7], gh[3]);
        }
        if (j > ka) {   // second step, row k
            const int k = j - 1, o = WALLS && wall >= 0 ? wall : k;   // row pulled, row written
            const int u = 7 + 5 * (k & 1);
            V2 ph, lin, nl, iph, t1, t2, t3, t4;
            take(u, t1, t2);
            take(u + 1, t3, t4);
            take(u + 2, ph, lin);
            take(u + 3, nl, iph);
            V2 R = ref_of(reinterpret_cast<const uint32_t&>(keep[(u + 4) * TWO_THREADS]));
            g[1] += t1;
            g[2] += t2;
            g[3] += t3;
            g[4] += t4;
            V2 rho, ur, uz, dT;
            Sums<V2> sm = sums2(f);
            recover_two(c, row_consts32(c, k), ph, lin, nl, sm, g, R, rho, ur, uz, dT);
            if (WALLS && (edge || o != k)) {
                const V2 Rf = R, iphf = iph;
                if (o != k) {
                    ph = ld_two<VEC>(phi + o * nz, la, lb);
                    R = ref_of(ld_ref<VEC>(c.tref + o * nz, la, lb));
                    porous_two(c, ph, lin, nl, iph);
                }
                wall_pair<!VEC>(c, k, o, ca, f, g, sm.m0, rho, ur, uz, dT, iphf, Rf, ph, R);
                sm = sums2(f);
            }
            collide_two(c, row_consts32(c, o), ph, lin, nl, iph, sm, f, g, R, rho, ur, uz, dT);
            float* __restrict__ Fo = B.f + o * nz;
            float* __restrict__ Go = B.g + o * nz;
            if (st0) {
#pragma unroll
                for (int i = 0; i < 9; ++i) st_two<VEC>(Fo + i * plane + ca, f[i], st1);
#pragma unroll
                for (int i = 0; i < 5; ++i) st_two<VEC>(Go + i * plane + ca, g[i], st1);
            }
        }
    }
}

}  // namespace lbm
