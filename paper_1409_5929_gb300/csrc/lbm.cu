// lbm.cu -- kernels and host runtime behind the C ABI of include/lbm.h.
//
// Axisymmetric D2Q9 MRT flow + D2Q5 temperature lattice Boltzmann step for porous
// media (Liu, He & Li, arXiv 1409.5929, Sec. 3-4) on one GB300 (sm_103a).
//
// Data layout in HBM (per handle):
//   state A, state B: 14 planes (f_0..f_8, g_0..g_4), each nr*nz elements, z fastest,
//                     plane stride padded to 64 elements; f planes in the storage
//                     type (FP32, FP16 or BF16), g planes in FP32, holding the
//                     deviations of lbm_physics.cuh.  A step reads one buffer and
//                     writes the other.
//   phi:              nr*nz porosity values (FP32).
//   tref:             nr*nz temperature references R(x) (FP16).
//   fref:             nr*nz flow references Q(x), 4 x FP16 each (16-bit storage).
//   macro snapshots, reduction scratch, staging: only for diagnostics.
//
// A step in two buffers is one launch that holds its boundary nodes (FP32: lbm_f32.cu, on small and
// large grids several steps per launch; 16-bit storage: lbm_16.cu), except
//   k_bulk_stage + k_wall   16-bit storage on large grids: every non-wall node (pull, Eq. 22, 33;
//           recovery, Eq. 26-30, 38; collision, Eq. 21-24, 33-37; store), row sources staged in
//           shared memory; then every wall node (rebuild from the interior neighbour by
//           non-equilibrium extrapolation, Sec. 4, ref. [47], collision with u = 0 and the
//           wall temperature), one thread each;
//   k_bulk + k_wall         one node per thread: in-place storage (the wall kernel first), FP32
//           storage with the discrete heater, and grids beyond 32-bit indices.
// Both kernels of a pair read only the source buffer and write disjoint nodes of the destination.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda.h>
#include <cuda_runtime.h>

#include <array>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/lbm.h"
#include "lbm_16.h"
#include "lbm_f32.h"
#include "lbm_lists.h"
#include "lbm_nodes.cuh"
#include "lbm_pair.cuh"
#include "lbm_physics.cuh"

using namespace lbm;

// One thread per column segment of RPT rows: the column's index arithmetic, the
// kernel-argument loads and the class checks are shared by RPT nodes.
// I: index type; 32-bit when the state buffer holds fewer than 2^31 elements.
// Resident blocks of 128 threads per SM the register allocation must allow (0: no
// constraint).  16-bit flow storage is issue-bound: ten blocks (48 registers) beat the
// compiler's nine (measured 0.5303 vs 0.5425 ms at 4096 x 8192); FP32 is bandwidth-bound
// and does best with the compiler's own allocation (56 registers, 0.6079 ms; 0.6119 with
// nine blocks required, 0.6376 with ten).
// In place with 16-bit storage (one node per thread, shifted reads or stores): eight blocks
// (64 registers) measured 0.693 ms at 4096 x 8192 against 0.716 with nine and 0.737 with
// ten (48 registers, 36 bytes spilled).
#ifndef LBM_INPLACE16_MIN_BLOCKS
#define LBM_INPLACE16_MIN_BLOCKS 8
#endif
template <int STO, int LIN = LAY_N>
constexpr int bulk_min_blocks() { return STO == LBM_F32 ? 0 : (LIN == LAY_N ? 10 : LBM_INPLACE16_MIN_BLOCKS); }

template <int STO, typename I, int RPT, int LIN = LAY_N, int LOUT = LAY_N>
__global__ void __launch_bounds__(BULK_THREADS, bulk_min_blocks<STO, LIN>()) k_bulk(const Consts<float> c, const Buf<STO> A, const Buf<STO> B,
                                                       const typename St<STO>::P* __restrict__ phi, I plane) {
    const int kz = blockIdx.x * BULK_THREADS + threadIdx.x;
    if (kz >= c.nz) return;
    update_column<STO, I, LIN, LOUT>(c, A, B, phi, plane, blockIdx.y * RPT, RPT, kz);
}

#ifndef LBM_STAGE_MIN_BLOCKS
#define LBM_STAGE_MIN_BLOCKS 6
#endif
template <int STO, int RPT, bool ALN>
__global__ void __launch_bounds__(BULK_THREADS, LBM_STAGE_MIN_BLOCKS) k_bulk_stage(const Consts<float> c, const Buf<STO> A, const Buf<STO> B,
                                                             const float* __restrict__ phi, int plane, int spin,
                                                             int* __restrict__ status) {
    __shared__ PairStage<BULK_THREADS> sb;
    stage_block<STO, BULK_THREADS, ALN>(c, A, B, phi, plane, blockIdx.y * RPT, RPT, blockIdx.x * 2 * BULK_THREADS, spin,
                                        status, sb);
}

// The staged kernel keeps sizeof(PairStage<BULK_THREADS>) (30.7 KB) of shared memory per
// block; at LBM_STAGE_MIN_BLOCKS blocks per SM that needs the largest shared-memory carveout.
template <int STO>
static cudaError_t stage_carveout() {
    cudaError_t e = cudaFuncSetAttribute(k_bulk_stage<STO, BULK_RPT, true>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         (int)cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_bulk_stage<STO, BULK_RPT, false>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared);
    return e;
}

// Wall nodes; LIN / LOUT: layouts read and written (in-place storage alternates S and L).
template <int STO, int LIN = LAY_N, int LOUT = LAY_N>
__global__ void k_wall(const Consts<float> c, const Buf<STO> A,
                       const Buf<STO> B, const typename St<STO>::P* __restrict__ phi,
                       int64_t plane, int count) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= count) return;
    int kr, kz;
    wall_node(c.geometry, c.nr, c.nz, t, kr, kz);
    const int cls = node_class(c.geometry, c.nr, c.nz, kr, kz);
    float fh[9], gh[5], m0, rho, urb, uzb, dTb, refb;
    wall_state<STO, float, LIN>(c, A, phi, plane, cls, kr, kz, fh, gh, m0, rho, urb, uzb, dTb, refb);
    const int64_t n = (int64_t)kr * c.nz + kz;
    const float r = c.r0 + float(kr), ph = ldv(phi + n);
    float lin, nl, iph;
    porous(c, ph, lin, nl, iph);
    collide(c, r, rcp_acc(r), ph, lin, nl, iph, fh, gh, refb, m0, rho, urb, uzb, dTb);
    store<STO, float, int64_t, LOUT>(c, B, plane, kr, kz, n, fh, gh);
}

// Fields of a state at every node (NULL outputs skipped).
template <int STO, int LAY = LAY_N>
__global__ void k_moments(const Consts<float> c, const Buf<STO> A,
                          const typename St<STO>::P* __restrict__ phi, int64_t plane, float* rho_o, float* ur_o,
                          float* uz_o, float* T_o) {
    const int kz = blockIdx.x * blockDim.x + threadIdx.x;
    const int kr = blockIdx.y;
    if (kz >= c.nz) return;
    const int cls = node_class(c.geometry, c.nr, c.nz, kr, kz);
    const int64_t n = (int64_t)kr * c.nz + kz;
    float fh[9], gh[5], m0, rho, ur = 0.f, uz = 0.f, dT, ref;
    if (is_wall(cls)) {
        wall_state<STO, float, LAY>(c, A, phi, plane, cls, kr, kz, fh, gh, m0, rho, ur, uz, dT, ref);
    } else {
        pull<STO, float, int64_t, LAY>(c, A, plane, kr, kz, fh, gh, ref);
        const float r = c.r0 + float(kr), ph = ldv(phi + n);
        float lin, nl, iph;
        porous(c, ph, lin, nl, iph);
        recover(c, r, rcp_acc(r), ph, lin, nl, fh, gh, ref, m0, rho, ur, uz, dT);
    }
    if (rho_o) rho_o[n] = rho;
    if (ur_o) ur_o[n] = ur;
    if (uz_o) uz_o[n] = uz;
    if (T_o) T_o[n] = (c.T0 + ref) + dT;
}

// Start state (FP64 arithmetic, one launch per initialisation): pre-collision
// f = M^-1(m_eq - S/2) at rho = 1 (Eq. 19-20, 24), g = g_eq(T, u) (Eq. 35), then one
// collision at the node.  Cold start: T = T0 + noise * U(-1, 1) from SplitMix64.
__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t n) {
    uint64_t z = seed + (n + 1) * 0x9e3779b97f4a7c15ULL;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    return z ^ (z >> 31);
}

__device__ __forceinline__ double start_T(const Consts<double>& c, const float* T_in, double noise, uint64_t seed,
                                          int64_t n) {
    if (T_in) return (double)T_in[n];
    const double u01 = (double)(splitmix64(seed, (uint64_t)n) >> 11) * (1.0 / 9007199254740992.0);
    return c.T0 + noise * (2 * u01 - 1);
}

template <int STO>
__global__ void k_init(const Consts<double> c, const Buf<STO> B,
                       const typename St<STO>::P* __restrict__ phi, int64_t plane, const float* ur_in,
                       const float* uz_in, const float* T_in, double noise, uint64_t seed, __half* __restrict__ tref,
                       uint2* __restrict__ fref, int inplace) {
    const int kz = blockIdx.x * blockDim.x + threadIdx.x;
    const int kr = blockIdx.y;
    if (kz >= c.nz) return;
    const int64_t n = (int64_t)kr * c.nz + kz;
    const int cls = node_class(c.geometry, c.nr, c.nz, kr, kz);
    const double r = c.r0 + kr, inv_r = 1.0 / r;
    double T = start_T(c, T_in, noise, seed, n), ur = 0, uz = 0;
    if (cls == WALL_IN && c.heater) {
        int fr, fz;
        fluid_neighbour(c.geometry, c.nr, c.nz, cls, kr, kz, fr, fz);
        T = start_T(c, T_in, noise, seed, (int64_t)fr * c.nz + fz);
    } else if (cls == WALL_IN) T = c.T_hot;
    else if (cls == WALL_OUT) T = c.T_cold;
    else if (cls == INLET) {
        T = c.T_hot;
        uz = c.u_in;
    } else if (cls == BOTTOM || cls == TOP || cls == OUTLET) {
        int fr, fz;
        fluid_neighbour(c.geometry, c.nr, c.nz, cls, kr, kz, fr, fz);
        T = start_T(c, T_in, noise, seed, (int64_t)fr * c.nz + fz);
    } else if (ur_in && uz_in) {
        ur = ur_in[n];
        uz = uz_in[n];
    }
    const double ph = (double)ldv(phi + n);
    double lin, nl, iphi;
    porous(c, ph, lin, nl, iphi);
    const double um = sqrt(ur * ur + uz * uz);
    const double Fr = -ph * (lin + nl * um) * ur;
    const double Ftr = Fr + cs2<double>() * (1 - c.two_taum * ur * inv_r) * inv_r;
    const double Ftz = -ph * (lin + nl * um) * uz + ph * (c.gbeta * (T - c.T0) + c.az);
    const double u2 = ur * ur + uz * uz;
    // deviation moments of f = M^-1 (m_eq - S/2) at rho = 1 (S_3 without its rest c_s^2)
    const double S1 = 6 * r * (ur * Ftr + uz * Ftz) * iphi, S5 = r * Ftz;
    const double S3 = r * Fr - cs2<double>() * c.two_taum * ur * inv_r;
    const double S7 = 2 * r * (ur * Ftr - uz * Ftz) * iphi, S8 = r * (ur * Ftz + uz * Ftr) * iphi;
    const double q = 3 * r * u2 * iphi;
    const double mpre[9] = {0.0,
                            q - 0.5 * S1,
                            -q + 0.5 * S1,
                            r * ur - 0.5 * S3,
                            -r * ur + 0.5 * S3,
                            r * uz - 0.5 * S5,
                            -r * uz + 0.5 * S5,
                            r * (ur * ur - uz * uz) * iphi - 0.5 * S7,
                            r * ur * uz * iphi - 0.5 * S8};
    double fh[9], gh[5];
    minv(mpre, fh);
    // reference offset R(x) = T - T0 in FP16; gh relative to T0 + R(x)
    const __half Rh = __float2half_rn(fminf(fmaxf((float)(T - c.T0), -60000.f), 60000.f));
    if constexpr (!has_fref<STO>()) tref[n] = Rh;
    const double ref = (double)__half2float(Rh);
    const double dTs = T - c.T0 - ref;
    gh[0] = 0.6 * dTs;
    gh[1] = 0.1 * dTs + 0.5 * T * ur;
    gh[2] = 0.1 * dTs + 0.5 * T * uz;
    gh[3] = 0.1 * dTs - 0.5 * T * ur;
    gh[4] = 0.1 * dTs - 0.5 * T * uz;
    double m0, rho, u_r = ur, u_z = uz, dT;   // boundary nodes keep their start velocity
    if (is_wall(cls)) {
        m0 = ((fh[0] + fh[1]) + (fh[2] + fh[3])) + ((fh[4] + fh[5]) + (fh[6] + fh[7])) + fh[8];
        rho = 1 + m0 * inv_r;
        dT = dTs;
    } else {
        recover(c, r, inv_r, ph, lin, nl, fh, gh, ref, m0, rho, u_r, u_z, dT);
    }
    collide(c, r, inv_r, ph, lin, nl, iphi, fh, gh, ref, m0, rho, u_r, u_z, dT);
    if constexpr (has_fref<STO>()) {
        // the start state's own flow reference: the moments of its deviations
        double A = 0, Jr = 0, Jz = 0;
        for (int i = 0; i < 9; ++i) {
            A += fh[i];
            Jr += ex9(i) * fh[i];
            Jz += ez9(i) * fh[i];
        }
        const uint2 qw = fref_make((float)A, (float)Jr, (float)Jz, Rh);
        fref[n] = qw;
        const Qf q = fref_unpack(qw);
        for (int i = 0; i < 9; ++i)
            stv(B.f + (inplace ? opp9(i) : i) * plane + n, (float)(fh[i] - (double)fref_delta(i, q)));
    } else {
        for (int i = 0; i < 9; ++i) stv(B.f + (inplace ? opp9(i) : i) * plane + n, (float)fh[i]);
    }
    // in-place storage starts in layout S: population i in slot opp(i) of its own node
    for (int i = 0; i < 5; ++i) stv(B.g + (inplace ? opp9(i) : i) * plane + n, (float)gh[i]);
}

template <int STO> __device__ __forceinline__ typename St<STO>::P mkp(float v);
template <> __device__ __forceinline__ float mkp<LBM_F32>(float v) { return v; }
template <> __device__ __forceinline__ float mkp<LBM_F16>(float v) { return v; }
template <> __device__ __forceinline__ float mkp<LBM_BF16>(float v) { return v; }

// Porosity upload: validate (0 < phi <= 1) and convert to the storage type.
__device__ __forceinline__ unsigned int bad_phi(float v) { return !(v > 0.f && v <= 1.f); }

// Porosity upload: count of values outside (0, 1] and conversion to the storage type.
// Grid-stride; 16-byte loads when src is 16-byte aligned (vec != 0), then the ragged tail
// one value at a time.
template <int STO>
__global__ void k_phi(const float* __restrict__ src, typename St<STO>::P* __restrict__ dst, int64_t n, int vec,
                      unsigned int* bad) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n4 = vec ? n / 4 : 0;
    unsigned int cnt = 0;
    for (int64_t q = t; q < n4; q += stride) {
        const float4 v = reinterpret_cast<const float4*>(src)[q];
        cnt += bad_phi(v.x) + bad_phi(v.y) + bad_phi(v.z) + bad_phi(v.w);
        dst[4 * q] = mkp<STO>(v.x);
        dst[4 * q + 1] = mkp<STO>(v.y);
        dst[4 * q + 2] = mkp<STO>(v.z);
        dst[4 * q + 3] = mkp<STO>(v.w);
    }
    for (int64_t i = 4 * n4 + t; i < n; i += stride) {
        const float v = src[i];
        cnt += bad_phi(v);
        dst[i] = mkp<STO>(v);
    }
    if (cnt) atomicAdd(bad, cnt);
}

// Two result values written into mapped host memory by the kernel itself (no copy-engine
// transfer for 16 bytes).
__global__ void k_put2(const double* __restrict__ src, double* dst, int skip_first) {
    const int i = threadIdx.x;
    if (i < 2 && !(skip_first && i == 0)) dst[i] = src[i];
}

// Range check alone (FP32 storage: the checked staging buffer becomes the field); src is a
// staging buffer (cudaMalloc, 16-byte aligned).
__global__ void k_phi_check(const float* __restrict__ src, int64_t n, unsigned int* bad) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n4 = n / 4;
    unsigned int cnt = 0;
    for (int64_t q = t; q < n4; q += stride) {
        const float4 v = reinterpret_cast<const float4*>(src)[q];
        cnt += bad_phi(v.x) + bad_phi(v.y) + bad_phi(v.z) + bad_phi(v.w);
    }
    for (int64_t i = 4 * n4 + t; i < n; i += stride) cnt += bad_phi(src[i]);
    if (cnt) atomicAdd(bad, cnt);
}

// Blocks of 256 threads for the grid-stride porosity kernels over n values.
static unsigned int phi_blocks(int64_t n) {
    return (unsigned int)std::max<int64_t>(1, std::min<int64_t>((n / 4 + 255) / 256, 4096));
}

static int aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

template <int STO>
__global__ void k_phi_fill(typename St<STO>::P* __restrict__ dst, int64_t n, float v) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = mkp<STO>(v);
}

__global__ void k_node_class(int geometry, int nr, int nz, uint8_t* out) {
    const int kz = blockIdx.x * blockDim.x + threadIdx.x;
    const int kr = blockIdx.y;
    if (kz < nz) out[(int64_t)kr * nz + kz] = (uint8_t)node_class(geometry, nr, nz, kr, kz);
}

// ----------------------------------------------------- FP64 reductions --
// Block sum of NV doubles per thread (warp shuffles, then shared memory).
template <int NV>
__device__ __forceinline__ void block_sum(double* v, double* out_if_thread0) {
    __shared__ double sh[32][NV];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int j = 0; j < NV; ++j)
        for (int o = 16; o > 0; o >>= 1) v[j] += __shfl_down_sync(0xffffffffu, v[j], o);
    if (lane == 0)
        for (int j = 0; j < NV; ++j) sh[warp][j] = v[j];
    __syncthreads();
    if (warp == 0) {
        const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            double x = lane < nw ? sh[lane][j] : 0.0;
            for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
            if (lane == 0) out_if_thread0[j] = x;
        }
    }
}

// Residual partials over nodes: |du|^2, |u|^2, dT^2, T^2 on non-wall nodes, mass
// r * rho on all nodes, and a count of non-finite values; one row of 6 per block.
constexpr int RES_NV = 6;
__global__ void k_resid_partial(int geometry, int nr, int nz, double r0, const float* __restrict__ cur,
                                const float* __restrict__ prev, int64_t fstride, double* __restrict__ partials) {
    double v[RES_NV] = {0, 0, 0, 0, 0, 0};
    const int64_t N = (int64_t)nr * nz;
    for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (int64_t)gridDim.x * blockDim.x) {
        const int kr = (int)(n / nz), kz = (int)(n - (int64_t)kr * nz);
        const float rho = cur[n], ur = cur[fstride + n], uz = cur[2 * fstride + n], T = cur[3 * fstride + n];
        if (!isfinite(rho) || !isfinite(ur) || !isfinite(uz) || !isfinite(T)) v[5] += 1;
        v[4] += (r0 + kr) * (double)rho;
        if (is_wall(node_class(geometry, nr, nz, kr, kz))) continue;
        const double a = (double)ur - prev[fstride + n], b = (double)uz - prev[2 * fstride + n];
        const double d = (double)T - prev[3 * fstride + n];
        v[0] += a * a + b * b;
        v[1] += (double)ur * ur + (double)uz * uz;
        v[2] += d * d;
        v[3] += (double)T * T;
    }
    double out[RES_NV];
    block_sum<RES_NV>(v, out);
    if (threadIdx.x == 0)
        for (int j = 0; j < RES_NV; ++j) partials[blockIdx.x * RES_NV + j] = out[j];
}

__global__ void k_sum_rows(const double* __restrict__ partials, int rows, double* __restrict__ result) {
    double v[RES_NV] = {0, 0, 0, 0, 0, 0};
    for (int b = threadIdx.x; b < rows; b += blockDim.x)
        for (int j = 0; j < RES_NV; ++j) v[j] += partials[b * RES_NV + j];
    double out[RES_NV];
    block_sum<RES_NV>(v, out);
    if (threadIdx.x == 0)
        for (int j = 0; j < RES_NV; ++j) result[j] = out[j];
}

// Temperature of node (kr, kz) of a state: wall temperature, the interior
// neighbour's T on adiabatic walls, else sum of the pulled g (Eq. 38), in FP64.
template <int STO, int LAY = LAY_N>
__device__ double node_T(const Consts<float>& c, const Buf<STO> A, int64_t plane, int kr,
                         int kz) {
    const int cls = node_class(c.geometry, c.nr, c.nz, kr, kz);
    if (cls == WALL_IN || cls == INLET) return (double)c.T_hot;
    if (cls == WALL_OUT) return (double)c.T_cold;
    if (cls == BOTTOM || cls == TOP || cls == OUTLET) {
        int fr, fz;
        fluid_neighbour(c.geometry, c.nr, c.nz, cls, kr, kz, fr, fz);
        kr = fr;
        kz = fz;
    }
    float fh[9], gh[5], ref;
    pull<STO, float, int64_t, LAY>(c, A, plane, kr, kz, fh, gh, ref);
    return (double)c.T0 + (double)ref + (((double)gh[0] + gh[1]) + ((double)gh[2] + gh[3]) + gh[4]);
}

// Eq. 42 for both walls: one-sided second-order dT/dr, trapezoid in z.  One column per
// thread, a partial sum per block; k_nusselt_final adds the partials in block order.
template <int STO, int LAY = LAY_N>
__global__ void __launch_bounds__(128) k_nusselt(const Consts<float> c, const Buf<STO> A, int64_t plane,
                                                 double* __restrict__ partials) {
    double v[2] = {0, 0};
    for (int kz = blockIdx.x * blockDim.x + threadIdx.x; kz < c.nz; kz += gridDim.x * blockDim.x) {
        const double wz = (kz == 0 || kz == c.nz - 1) ? 0.5 : 1.0;
        const double t0 = node_T<STO, LAY>(c, A, plane, 0, kz), t1 = node_T<STO, LAY>(c, A, plane, 1, kz);
        const double t2 = node_T<STO, LAY>(c, A, plane, 2, kz);
        const double u0 = node_T<STO, LAY>(c, A, plane, c.nr - 1, kz);
        const double u1 = node_T<STO, LAY>(c, A, plane, c.nr - 2, kz);
        const double u2 = node_T<STO, LAY>(c, A, plane, c.nr - 3, kz);
        v[0] += wz * (-3 * t0 + 4 * t1 - t2) * 0.5;
        v[1] += wz * (3 * u0 - 4 * u1 + u2) * 0.5;
    }
    double out[2];
    block_sum<2>(v, out);
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = out[0];
        partials[2 * blockIdx.x + 1] = out[1];
    }
}

__global__ void __launch_bounds__(256) k_nusselt_final(const double* __restrict__ partials, int blocks, double ri,
                                                       double ro, double H, double dTw, double* __restrict__ result) {
    double v[2] = {0, 0};
    for (int b = threadIdx.x; b < blocks; b += blockDim.x) {
        v[0] += partials[2 * b];
        v[1] += partials[2 * b + 1];
    }
    double out[2];
    block_sum<2>(v, out);
    if (threadIdx.x == 0) {
        result[0] = -ri * out[0] / (H * dTw);
        result[1] = -ro * out[1] / (H * dTw);
    }
}

// Eq. 40 per column for the pipe with inlet and outlet: Nu(z) = D (dT/dr)_w / (T_w - T_b)
// with the mixing-cup T_b = int u_z r T dr / int u_z r dr (trapezoid on r = 0, r0, r0 + 1,
// ..., r_i; the integrand is 0 at r = 0) and the one-sided second-order wall derivative.
// uz, T: field planes (row stride nz).  One thread per column, FP64.
__global__ void k_pipe_nusselt(int nr, int nz, double r0, const float* __restrict__ uz, const float* __restrict__ T,
                               double* __restrict__ nu) {
    const int kz = blockIdx.x * blockDim.x + threadIdx.x;
    if (kz >= nz) return;
    double num = 0.25 * (r0 * (double)uz[kz] * (double)T[kz]), den = 0.25 * (r0 * (double)uz[kz]);
    for (int k = 0; k + 1 < nr; ++k) {
        const int64_t a = (int64_t)k * nz + kz, b = a + nz;
        const double ra = r0 + k, rb = r0 + k + 1;
        num += 0.5 * (ra * (double)uz[a] * (double)T[a] + rb * (double)uz[b] * (double)T[b]);
        den += 0.5 * (ra * (double)uz[a] + rb * (double)uz[b]);
    }
    const double Tw = T[(int64_t)(nr - 1) * nz + kz];
    const double dTdr = (3 * Tw - 4 * (double)T[(int64_t)(nr - 2) * nz + kz] + (double)T[(int64_t)(nr - 3) * nz + kz]) / 2;
    nu[kz] = 2 * (r0 + (nr - 1)) * dTdr / (Tw - num / den);
}

// Eq. 43-44 for the discrete heater: Nu(z) = dT / (T_h(z) - T_o) at the heated inner-wall
// columns hz0..hz1 (corners excluded unless z is periodic), NaN elsewhere, and the mean
// over the heated columns.  Th: the inner-wall row of the T field.  One block, FP64.
__global__ void __launch_bounds__(256) k_heater_nusselt(int nz, int hz0, int hz1, int periodic, double dT, double To,
                                                        const float* __restrict__ Th, double* __restrict__ nu_z,
                                                        double* __restrict__ result) {
    double v[2] = {0, 0};
    for (int kz = threadIdx.x; kz < nz; kz += blockDim.x) {
        const bool heated = kz >= hz0 && kz <= hz1 && (periodic || (kz > 0 && kz < nz - 1));
        const double nu = heated ? dT / ((double)Th[kz] - To) : NAN;
        nu_z[kz] = nu;
        if (heated) {
            v[0] += nu;
            v[1] += 1;
        }
    }
    double out[2];
    block_sum<2>(v, out);
    if (threadIdx.x == 0) result[0] = out[1] > 0 ? out[0] / out[1] : NAN;
}

// Stokes stream function of the axisymmetric flow (|psi|max of Table 3):
// psi(r, z) = int_{r_s}^{r} r' u_z dr' so that r u_z = d psi/dr and, by Eq. 1,
// r u_r = -d psi/dz; r_s is the inner wall (annulus) or the axis (pipes, whose first
// panel runs from r = 0 to the first row at r0).  One thread per column walks the rows
// (each row's read is coalesced across the block), accumulating in FP64; every block
// writes the largest |psi| of its columns to block_max[blockIdx.x].
__global__ void __launch_bounds__(128) k_stream_function(int nr, int nz, double r0, int from_axis,
                                                         const float* __restrict__ uz, float* __restrict__ psi,
                                                         double* __restrict__ block_max) {
    const int kz = blockIdx.x * blockDim.x + threadIdx.x;
    double big = 0;
    if (kz < nz) {
        double prev = r0 * (double)uz[kz];
        double s = from_axis ? 0.5 * r0 * prev : 0.0;
        psi[kz] = (float)s;
        big = fabs(s);
        for (int k = 1; k < nr; ++k) {
            const int64_t n = (int64_t)k * nz + kz;
            const double cur = (r0 + k) * (double)uz[n];
            s += 0.5 * (prev + cur);
            prev = cur;
            psi[n] = (float)s;
            big = fmax(big, fabs(s));
        }
    }
    for (int o = 16; o > 0; o >>= 1) big = fmax(big, __shfl_down_sync(0xffffffffu, big, o));
    __shared__ double sh[4];
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = big;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x + 31) / 32; ++w) big = fmax(big, sh[w]);
        block_max[blockIdx.x] = big;
    }
}

// FP64 export of rows [row0, row0 + nrows): raw post-collision populations
// f_i = ft_i + r w_i + e_ir w_i / 2, g_i = gh_i + wT_i (T0 + R(x)), from the state in layout
// LAY (NaN for a population that layout does not keep).
template <int STO, int LAY = LAY_N>
__global__ void k_export(const Consts<float> c, const Buf<STO> A, int64_t plane, int row0,
                         int nrows, double r0, double T0, double* __restrict__ out) {
    const int kz = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (kz >= c.nz || j >= nrows) return;
    const int kr = row0 + j;
    const int64_t n = (int64_t)kr * c.nz + kz, m = (int64_t)j * c.nz + kz, P = (int64_t)nrows * c.nz;
    const double r = r0 + kr;
    const double wt[5] = {0.6, 0.1, 0.1, 0.1, 0.1};
    const double Tb = T0 + (double)tref_at<STO>(c, n);
    for (int i = 0; i < 9; ++i) {
        int64_t at;
        int slot;
        if (!own_slot<LAY, float, int64_t>(c, kr, kz, i, at, slot)) {
            out[i * P + m] = NAN;
            if (i < 5) out[(9 + i) * P + m] = NAN;
            continue;
        }
        double ref = 0.0;
        if constexpr (has_fref<STO>()) ref = (double)fref_delta(i, fref_unpack(c.fref[n]));
        out[i * P + m] = (double)ldv(A.f + slot * plane + at) + ref + (r + 0.5 * ex9(i)) * w9<double>(i);
        if (i < 5) out[(9 + i) * P + m] = (double)ldv(A.g + slot * plane + at) + wt[i] * Tb;
    }
}

// Reference refresh: R(x) <- FP16(R(x) + sum_i gh_i(x)), gh re-expressed against the
// new reference (gh_0 += d - 4 d/10, gh_1..4 += d/10 with d = R_old - R_new).  The
// populations, and every field they give, are unchanged up to rounding.
// Node (kr, kz) = n, state in layout LAY: the locations of its own populations (own_slot);
// a population the layout does not keep counts as a zero deviation (any R is a valid one).
template <int STO, int LAY, typename I>
__device__ __forceinline__ void rebase_thermal_node(const Consts<float>& c, const Buf<STO>& A, I plane, int kr,
                                                    int kz, I n, __half* __restrict__ tref) {
    float g[5];
    I at[5];
    int slot[5];
    bool kept[5], all = true;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        kept[i] = own_slot<LAY, float, I>(c, kr, kz, i, at[i], slot[i]);
        all = all && kept[i];
        g[i] = kept[i] ? ldv(A.g + slot[i] * plane + at[i]) : 0.f;
    }
    // a boundary node whose outgoing populations the layout dropped keeps its reference
    // (the kept ones do not sum to its temperature)
    if (!all) return;
    const float r_old = __half2float(tref[n]);
    const float t = r_old + (((g[0] + g[1]) + (g[2] + g[3])) + g[4]);
    const __half h = __float2half_rn(fminf(fmaxf(t, -60000.f), 60000.f));
    const float d = r_old - __half2float(h), d1 = 0.1f * d;
    g[0] += d - 4.f * d1;
#pragma unroll
    for (int i = 1; i < 5; ++i) g[i] += d1;
#pragma unroll
    for (int i = 0; i < 5; ++i)
        stv(A.g + slot[i] * plane + at[i], g[i]);
    tref[n] = h;
}

template <int STO, int LAY = LAY_N>
__global__ void k_rebase(const Consts<float> c, const Buf<STO> A, int64_t plane, int64_t N, __half* __restrict__ tref) {
    if constexpr (has_ref<STO>()) {
        for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (int64_t)gridDim.x * blockDim.x)
            rebase_thermal_node<STO, LAY, int64_t>(c, A, plane, (int)(n / c.nz), (int)(n % c.nz), n, tref);
    }
}

// Reference refresh (16-bit storage) of node n: decode its flow populations with the old
// reference word (as the pull does), take the new A, J from their deviation moments and the
// new R from the node's temperature (as rebase_thermal_node does), re-express the thermal
// deviations against the new R and re-encode the flow populations against the new A, J.
// The populations, and every field they give, are unchanged up to the storage rounding of
// the re-encoded (now small) values.
template <int STO, int LAY, typename I>
__device__ __forceinline__ void rebase_16_node(const Consts<float>& c, const Buf<STO>& S, I plane, int kr, int kz,
                                               I n, uint2* __restrict__ fref) {
    const Qf q0 = fref_unpack(fref[n]);
    float d[9], g[5];
    I at[9];
    int slot[9];
    bool kept[9], all = true;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        kept[i] = own_slot<LAY, float, I>(c, kr, kz, i, at[i], slot[i]);
        all = all && kept[i];
        d[i] = (kept[i] ? ldv(S.f + slot[i] * plane + at[i]) : 0.f) + fref_delta(i, q0);
        if (i < 5) g[i] = kept[i] ? ldv(S.g + slot[i] * plane + at[i]) : 0.f;
    }
    // a boundary node whose outgoing populations the layout dropped keeps its references:
    // the kept populations do not give its moments
    if (!all) return;
    const float a = ((d[0] + d[1]) + (d[2] + d[3])) + ((d[4] + d[5]) + (d[6] + d[7])) + d[8];
    const float jr = (d[1] - d[3]) + (d[5] - d[6]) + (d[8] - d[7]);
    const float jz = (d[2] - d[4]) + (d[5] + d[6]) - (d[7] + d[8]);
    const float t = q0.R + (((g[0] + g[1]) + (g[2] + g[3])) + g[4]);
    const __half h = __float2half_rn(fminf(fmaxf(t, -60000.f), 60000.f));
    const float dr = q0.R - __half2float(h), dr1 = 0.1f * dr;
    g[0] += dr - 4.f * dr1;
#pragma unroll
    for (int i = 1; i < 5; ++i) g[i] += dr1;
    const uint2 qw = fref_make(a, jr, jz, h);
    const Qf q1 = fref_unpack(qw);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        stv(S.f + slot[i] * plane + at[i], d[i] - fref_delta(i, q1));
        if (i < 5) stv(S.g + slot[i] * plane + at[i], g[i]);
    }
    fref[n] = qw;
}

template <int STO, int LAY = LAY_N>
__global__ void k_rebase_16(const Consts<float> c, const Buf<STO> S, int64_t plane, int64_t N,
                            uint2* __restrict__ fref) {
    if constexpr (has_fref<STO>()) {
        for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (int64_t)gridDim.x * blockDim.x)
            rebase_16_node<STO, LAY, int64_t>(c, S, plane, (int)(n / c.nz), (int)(n % c.nz), n, fref);
    }
}

// ------------------------------------------------------------ host runtime --
static thread_local std::string g_err;

static int fail(int code, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

#define CK(call)                                                                                   \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess) {                                                                   \
            (void)cudaGetLastError();                                                              \
            return fail(e_ == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA, "%s: %s (%s:%d)", \
                        #call, cudaGetErrorString(e_), __FILE__, __LINE__);                        \
        }                                                                                          \
    } while (0)

struct lbm_handle {
    lbm_params p;
    lbm_info info;
    Consts<float> cf;
    Consts<double> cd;
    int device = 0;
    int sms = 0;             // multiprocessors of the device
    cudaStream_t stream = nullptr;
    int64_t plane = 0;       // elements per plane (padded)
    int64_t N = 0;           // nr * nz
    void* buf[2] = {nullptr, nullptr};
    int cur = 0;             // buffer holding the current state
    void* phi = nullptr;
    __half* tref = nullptr;  // per-node reference offset R(x) of the thermal deviations
    uint2* fref = nullptr;   // per-node flow reference Q(x) (16-bit storage)
    int64_t since_rebase = 0;  // steps since the last flow-reference refresh
    int aa = 0;              // 1: in-place storage (one state buffer, layouts S and L alternate)
    int aa_odd = 0;          // in-place: 0 = state in layout S, 1 = in layout L
    float* fstage = nullptr; // N floats: porosity / init field upload
    // lbm_set_porosity_async: its own copy stream, two staging buffers (the upload into one
    // overlaps the steps that read the other), events and an error count
    cudaStream_t copy_stream = nullptr;
    float* astage[2] = {nullptr, nullptr};
    cudaEvent_t copied[2] = {nullptr, nullptr}, consumed[2] = {nullptr, nullptr};
    int astage_i = 0;
    int phi_pending = -1;           // staging buffer uploaded but not yet converted into phi
    unsigned int* bad_async = nullptr;
    float* mac = nullptr;    // two snapshots of 4 planes: rho, ur, uz, T
    int64_t mstride = 0;
    double* partials = nullptr;
    int pblocks = 0;
    double* result = nullptr;   // 8 doubles
    unsigned int* bad = nullptr;
    uint8_t* cls = nullptr;
    bool timing = false;
    std::vector<cudaEvent_t> ev;   // (bulk start, bulk end, wall start, wall end) per timed step
    int* wait_status = nullptr;    // 16-bit storage: LBM_ERR_TIMEOUT once a bounded wait of the staged kernel ran out
    int spin = STAGE_SPIN;         // try_wait rounds of its per-row waits
    bool limit_set = false;        // by lbm_set_wait_limit, to any value
    int stage = 1;                 // 16-bit: the staged bulk kernel where it applies (lbm_set_staging)
    Plan32 plan = {};              // launches of several steps (FP32 storage, two buffers)
    Consts32 c32;
    Step16 s16;                    // one launch per step (16-bit storage, two buffers)
    bool step16 = false;
};

static int derive(const lbm_params* p, lbm_info* o, Consts<double>* cd) {
    memset(o, 0, sizeof(*o));
    if (!p) return fail(LBM_ERR_INVALID, "params is NULL");
    if (p->nr < 3 || p->nz < 3) return fail(LBM_ERR_INVALID, "grid %d x %d: need nr, nz >= 3", p->nr, p->nz);
    if (p->nr > 65535) return fail(LBM_ERR_INVALID, "nr = %d exceeds 65535", p->nr);
    if (p->geometry < 0 || p->geometry > 3) return fail(LBM_ERR_INVALID, "unknown geometry %d", p->geometry);
    if (p->storage < 0 || p->storage > 2) return fail(LBM_ERR_INVALID, "unknown storage %d", p->storage);
    if (p->collision != LBM_MRT && p->collision != LBM_BGK)
        return fail(LBM_ERR_INVALID, "unknown collision %d", p->collision);
    if (p->inplace != 0 && p->inplace != 1) return fail(LBM_ERR_INVALID, "inplace must be 0 or 1");
    if (!(p->J > 0) || !(p->lambda > 0) || !(p->Pr > 0))
        return fail(LBM_ERR_INVALID, "J, lambda and Pr must be positive");
    if (!(p->eps_mean > 0 && p->eps_mean <= 1)) return fail(LBM_ERR_INVALID, "eps_mean %g outside (0, 1]", p->eps_mean);
    const double cs = std::sqrt(1.0 / 3.0);
    if (p->geometry == PIPE_PERIODIC_Z || p->geometry == PIPE_INFLOW) {
        o->r0 = 0.5;
        o->L = (p->nr - 1) + 0.5;
    } else {
        if (!(p->radius_ratio > 1)) return fail(LBM_ERR_INVALID, "radius_ratio %g must exceed 1", p->radius_ratio);
        o->L = p->nr - 1;
        o->r0 = o->L / (p->radius_ratio - 1);
    }
    o->H = p->nz - 1;
    const double dTw = p->T_hot - p->T_cold;
    if (p->tau_nu > 0) {
        o->tau_nu = p->tau_nu;
        o->Ma = p->Ra > 0 ? (o->tau_nu - 0.5) * cs * std::sqrt(p->Ra) / (p->J * o->L * std::sqrt(p->Pr)) : 0.0;
    } else {
        if (!(p->Ra > 0)) return fail(LBM_ERR_INVALID, "Ra must be positive when tau_nu is not given");
        o->Ma = p->Ma;
        o->tau_nu = 0.5 + p->Ma * p->J * o->L * std::sqrt(p->Pr) / (cs * std::sqrt(p->Ra));   // Eq. 39
    }
    if (!(o->tau_nu > 0.5)) return fail(LBM_ERR_INVALID, "tau_nu = %g must exceed 1/2", o->tau_nu);
    o->tau_T = (1.0 / 3.0) * p->lambda * (o->tau_nu - 0.5) / (0.2 * p->J * p->Pr);            // Eq. 39
    o->nu_e = (o->tau_nu - 0.5) / 3.0;                                                           // Eq. 31
    o->nu = o->nu_e / p->J;
    if (p->Ra > 0) {
        if (dTw == 0) return fail(LBM_ERR_INVALID, "T_hot == T_cold with Ra > 0");
        const double U = o->Ma * cs;                                                             // Ma = U / c_s
        o->gbeta = U * U / (dTw * o->L);                                                         // U^2 = g beta dT L
    }
    if (p->heater_len > 0) {
        if (p->geometry != LBM_ANNULUS && p->geometry != LBM_ANNULUS_PERIODIC_Z)
            return fail(LBM_ERR_INVALID, "the discrete heater needs an annulus geometry");
        if (p->nr < 4) return fail(LBM_ERR_INVALID, "the discrete heater needs nr >= 4");
        if (!(p->heater_len <= 1)) return fail(LBM_ERR_INVALID, "heater_len %g exceeds 1 (l / H)", p->heater_len);
        if (!(p->heater_center >= 0 && p->heater_center <= 1))
            return fail(LBM_ERR_INVALID, "heater_center %g outside [0, 1] (h / H)", p->heater_center);
    }
    if (p->geometry == LBM_PIPE_INFLOW && !(p->u_in >= 0 && p->u_in < 0.5))
        return fail(LBM_ERR_INVALID, "u_in = %g: the inlet velocity must lie in [0, 1/2)", p->u_in);
    o->T0 = p->heater_len > 0 ? p->T_cold : 0.5 * (p->T_hot + p->T_cold);   // Sec. 4.4: T0 = T_o
    o->Kbar = p->Da * o->L * o->L;
    const int64_t N = (int64_t)p->nr * p->nz;
    // populations read and written, porosity, and the references each node's pull reads:
    // R(x) (FP16) with FP32 storage, the reference word (A, J_r, J_z, R; 4 x FP16) with 16-bit
    // storage
    o->bytes_per_step = N * (int64_t)(2 * (9 * f_size(p->storage) + 5 * g_size(p->storage)) + phi_size(p->storage) +
                                      (p->storage == LBM_F32 ? sizeof(__half) : sizeof(uint2)));
    if (cd) {
        Consts<double>& c = *cd;
        memset(&c, 0, sizeof(c));
        c.nr = p->nr;
        c.nz = p->nz;
        c.geometry = p->geometry;
        c.periodic = periodic_z(p->geometry) ? 1 : 0;
        c.porous_mode = !(p->Da > 0) ? 0 : (p->eps_mean >= 1 ? 1 : 2);
        c.ergun = p->F_eps < 0;
        c.r0 = o->r0;
        c.cs2tau = (o->tau_nu - 0.5) / 3.0;
        c.two_taum = 2 * (o->tau_nu - 0.5);
        c.s_e = 1.1;
        c.s_eps = 1.1;
        c.s_j = 1.0;
        c.s_q = 1.2;
        c.s_nu = 1.0 / o->tau_nu;
        if (p->collision == LBM_BGK)   // Sec. 3.1: every moment relaxes at 1/tau
            c.s_e = c.s_eps = c.s_j = c.s_q = c.s_nu;
        c.h_e = 1 - 0.5 * c.s_e;
        c.h_eps = 1 - 0.5 * c.s_eps;
        c.h_j = 1 - 0.5 * c.s_j;
        c.h_q = 1 - 0.5 * c.s_q;
        c.h_nu = 1 - 0.5 * c.s_nu;
        c.cs2_2tm = c.two_taum / 3.0;
        c.tauT = o->tau_T;
        c.wg_den = 1.0 / (o->tau_T + 0.5);
        c.gbeta = o->gbeta;
        c.T0 = o->T0;
        c.az = p->body_accel_z;
        c.u_in = p->u_in;
        if (p->heater_len > 0) {
            const double H = p->nz - 1, h = p->heater_center * H, half = 0.5 * p->heater_len * H;
            c.heater = 1;
            c.hz0 = (int)std::max(0.0, std::ceil(h - half));
            c.hz1 = (int)std::min(H, std::floor(h + half));
            c.hG = (p->T_hot - p->T_cold) / o->L;
        }
        // Eq. 8 coefficients (see porous()): 1/K(phi) = c_k (1 - phi)^2 / phi^3 with
        // c_k = eps_mean^3 / ((1 - eps_mean)^2 Da L^2), i.e. K(eps_mean) = Da L^2.
        const double em = p->eps_mean;
        const double F = p->F_eps > 0 ? p->F_eps : 0.0;
        if (c.porous_mode == 2) {
            const double ck = em * em * em / ((1 - em) * (1 - em) * o->Kbar);
            c.lin_coef = o->nu * ck;
            c.nl_coef = c.ergun ? 1.75 * std::sqrt(ck / 150.0) : F * std::sqrt(ck);
        } else if (c.porous_mode == 1) {
            c.lin_coef = o->nu / o->Kbar;
            c.nl_coef = c.ergun ? 1.75 * std::sqrt(1.0 / (150.0 * o->Kbar)) : F / std::sqrt(o->Kbar);
        }
        c.T_hot = p->T_hot;
        c.T_cold = p->T_cold;
    }
    return LBM_OK;
}

static Consts<float> to_float(const Consts<double>& d) {
    Consts<float> f;
    f.nr = d.nr; f.nz = d.nz; f.geometry = d.geometry; f.porous_mode = d.porous_mode; f.ergun = d.ergun; f.periodic = d.periodic;
    f.heater = d.heater; f.hz0 = d.hz0; f.hz1 = d.hz1; f.hG = (float)d.hG;
    f.r0 = (float)d.r0; f.cs2tau = (float)d.cs2tau; f.two_taum = (float)d.two_taum;
    f.s_e = (float)d.s_e; f.s_eps = (float)d.s_eps; f.s_j = (float)d.s_j; f.s_q = (float)d.s_q; f.s_nu = (float)d.s_nu;
    f.h_e = (float)d.h_e; f.h_eps = (float)d.h_eps; f.h_j = (float)d.h_j; f.h_q = (float)d.h_q; f.h_nu = (float)d.h_nu;
    f.cs2_2tm = (float)d.cs2_2tm;
    f.tauT = (float)d.tauT; f.wg_den = (float)d.wg_den; f.gbeta = (float)d.gbeta; f.T0 = (float)d.T0;
    f.az = (float)d.az; f.lin_coef = (float)d.lin_coef; f.nl_coef = (float)d.nl_coef;
    f.T_hot = (float)d.T_hot; f.T_cold = (float)d.T_cold;
    f.u_in = (float)d.u_in;
    f.tref = d.tref;
    return f;
}

// Work that reads or writes the porosity field first waits for an asynchronous upload.
static dim3 grid2d(const lbm_handle* h, int threads) {
    return dim3((unsigned)((h->p.nz + threads - 1) / threads), (unsigned)h->p.nr);
}

// Dispatch a templated launch on the storage type.
#define DISPATCH_STO(sto, ...)                      \
    switch (sto) {                                  \
        case LBM_F32: { constexpr int S_ = LBM_F32; __VA_ARGS__; } break;  \
        case LBM_F16: { constexpr int S_ = LBM_F16; __VA_ARGS__; } break;  \
        default: { constexpr int S_ = LBM_BF16; __VA_ARGS__; } break;      \
    }

// Dispatch on the two 16-bit storage types.
#define DISPATCH_STO16(sto, ...)                                           \
    switch (sto) {                                                         \
        case LBM_F16: { constexpr int S_ = LBM_F16; __VA_ARGS__; } break;  \
        default: { constexpr int S_ = LBM_BF16; __VA_ARGS__; } break;      \
    }

// Layout of a state: A/B buffers, or in-place after an even (S) or odd (L) number of steps.
#define DISPATCH_LAY(lay, ...)                                             \
    switch (lay) {                                                         \
        case LAY_S: { constexpr int L_ = LAY_S; __VA_ARGS__; } break;      \
        case LAY_L: { constexpr int L_ = LAY_L; __VA_ARGS__; } break;      \
        default: { constexpr int L_ = LAY_N; __VA_ARGS__; } break;         \
    }

// rows per thread of the batched kernels: 1, 2 or 4 (the values the tuner tries)
#define DISPATCH_RPT(rpt, ...)                                             \
    switch (rpt) {                                                         \
        case 4: { constexpr int R_ = 4; __VA_ARGS__; } break;              \
        case 2: { constexpr int R_ = 2; __VA_ARGS__; } break;              \
        default: { constexpr int R_ = 1; __VA_ARGS__; } break;             \
    }

template <int STO> static Buf<STO> bufp(const lbm_handle* h, int which) {
    Buf<STO> b;
    char* base = (char*)h->buf[which];
    b.f = (typename St<STO>::TF*)base;
    b.g = (typename St<STO>::TG*)(base + 9 * h->plane * f_size(STO));
    return b;
}
template <int STO> using PP = typename St<STO>::P;

static int wait_phi(lbm_handle* h) {
    if (h->phi_pending >= 0) {
        // the newest upload becomes the field: on the compute stream, after everything
        // queued before (which read the old field) and after its copy
        const int i = h->phi_pending;
        h->phi_pending = -1;
        CK(cudaStreamWaitEvent(h->stream, h->copied[i], 0));
        const unsigned blocks = phi_blocks(h->N);
        // the field is FP32 for every storage type: check the staging buffer and swap it with
        // the field; the old field becomes staging buffer i once the work queued before has
        // read it
        k_phi_check<<<blocks, 256, 0, h->stream>>>(h->astage[i], h->N, h->bad_async);
        void* old = h->phi;
        h->phi = h->astage[i];
        h->astage[i] = (float*)old;
        CK(cudaGetLastError());
        CK(cudaEventRecord(h->consumed[i], h->stream));
    }
    return LBM_OK;
}

extern "C" {

void lbm_params_default(lbm_params* p) {
    if (!p) return;
    memset(p, 0, sizeof(*p));
    p->nr = 48;
    p->nz = 96;
    p->geometry = LBM_ANNULUS;
    p->storage = LBM_F32;
    p->radius_ratio = 2.0;
    p->Ra = 1e3;
    p->Da = 1e-2;
    p->Pr = 1.0;
    p->J = 1.0;
    p->lambda = 1.0;
    p->Ma = 0.1;
    p->tau_nu = 0.0;
    p->F_eps = -1.0;
    p->eps_mean = 0.6;
    p->T_hot = 1.0;
    p->T_cold = 0.0;
    p->body_accel_z = 0.0;
    p->init_noise = 1e-3;
    p->seed = 1;
    p->heater_center = 0.5;
}

int lbm_derive(const lbm_params* p, lbm_info* out) {
    if (!out) return fail(LBM_ERR_INVALID, "out is NULL");
    return derive(p, out, nullptr);
}

int lbm_destroy(lbm_handle* h) {
    if (!h) return LBM_OK;
    cudaSetDevice(h->device);
    if (h->copy_stream) cudaStreamSynchronize(h->copy_stream);   // an upload may still write phi
    if (h->stream) cudaStreamSynchronize(h->stream);
    for (void* b : h->buf) cudaFree(b);
    cudaFree(h->tref);
    cudaFree(h->fref);
    cudaFree(h->phi);
    cudaFree(h->fstage);
    if (h->copy_stream) cudaStreamDestroy(h->copy_stream);
    for (int i = 0; i < 2; ++i) {
        cudaFree(h->astage[i]);
        if (h->consumed[i]) cudaEventDestroy(h->consumed[i]);
        if (h->copied[i]) cudaEventDestroy(h->copied[i]);
    }
    cudaFree(h->bad_async);
    cudaFree(h->mac);
    cudaFree(h->partials);
    cudaFree(h->result);
    cudaFree(h->bad);
    cudaFree(h->cls);
    cudaFree(h->wait_status);
    for (auto e : h->ev)
        if (e) cudaEventDestroy(e);
    delete h;
    return LBM_OK;
}

static int launch_init(lbm_handle* h, const float* ur, const float* uz, const float* T) {
    if (int rc = wait_phi(h)) return rc;
    dim3 g = grid2d(h, 128);
    DISPATCH_STO(h->p.storage,
                 k_init<S_><<<g, 128, 0, h->stream>>>(h->cd, bufp<S_>(h, 0), (const PP<S_>*)h->phi, h->plane, ur, uz,
                                                      T, h->p.init_noise, h->p.seed, h->tref, h->fref, h->aa));
    CK(cudaGetLastError());
    h->cur = 0;
    h->aa_odd = 0;
    h->info.steps = 0;
    h->since_rebase = 0;
    return LBM_OK;
}

int lbm_create(const lbm_params* p, lbm_handle** out) {
    if (!out) return fail(LBM_ERR_INVALID, "out is NULL");
    *out = nullptr;
    lbm_handle* h = new lbm_handle();
    int rc = derive(p, &h->info, &h->cd);
    if (rc) { delete h; return rc; }
    h->p = *p;
    h->cf = to_float(h->cd);
    cudaError_t e = cudaGetDevice(&h->device);
    if (e != cudaSuccess) { delete h; return fail(LBM_ERR_CUDA, "cudaGetDevice: %s", cudaGetErrorString(e)); }
    e = cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, h->device);
    if (e != cudaSuccess) { delete h; return fail(LBM_ERR_CUDA, "cudaDeviceGetAttribute: %s", cudaGetErrorString(e)); }
    if (p->storage != LBM_F32) {
        e = p->storage == LBM_F16 ? stage_carveout<LBM_F16>() : stage_carveout<LBM_BF16>();
        if (e != cudaSuccess) { delete h; return fail(LBM_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e)); }
    }
    h->N = (int64_t)p->nr * p->nz;
    h->plane = (h->N + 63) / 64 * 64;
    h->mstride = h->plane;
    h->pblocks = 1024;
#define ALLOC(ptr, bytes)                                                       \
    do {                                                                        \
        cudaError_t e_ = cudaMalloc((void**)&(ptr), (bytes));                   \
        if (e_ != cudaSuccess) {                                                \
            (void)cudaGetLastError();                                           \
            lbm_destroy(h);                                                     \
            return fail(e_ == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA, \
                        "cudaMalloc(%zu bytes): %s", (size_t)(bytes), cudaGetErrorString(e_)); \
        }                                                                       \
    } while (0)
    h->aa = p->inplace;
    ALLOC(h->buf[0], state_bytes(p->storage, h->plane));
    if (!h->aa) ALLOC(h->buf[1], state_bytes(p->storage, h->plane));
    if (p->storage == LBM_F32) {
        ALLOC(h->tref, h->plane * sizeof(__half));
        h->cd.tref = h->tref;
        h->cf.tref = h->tref;
    } else {
        ALLOC(h->fref, h->plane * sizeof(uint2));
        h->cd.fref = h->fref;
        h->cf.fref = h->fref;
        ALLOC(h->wait_status, sizeof(int));
        e = cudaMemset(h->wait_status, 0, sizeof(int));
        if (e != cudaSuccess) { lbm_destroy(h); return fail(LBM_ERR_CUDA, "cudaMemset: %s", cudaGetErrorString(e)); }
    }
    ALLOC(h->phi, h->plane * phi_size(p->storage));
    ALLOC(h->partials, (size_t)h->pblocks * RES_NV * sizeof(double));
    ALLOC(h->result, 8 * sizeof(double));
    ALLOC(h->bad, sizeof(unsigned int));
#undef ALLOC
    // several steps per launch: FP32 storage in two buffers indexed with 32 bits; the discrete
    // heater's wall reads a second row inward, which those kernels do not carry
    if (p->storage == LBM_F32 && !h->aa && !h->cf.heater && 14 * h->plane < ((int64_t)1 << 31)) {
        h->c32 = consts32(h->cd, h->cf);
        e = plan32(h->p, h->sms, &h->plan);
        if (e != cudaSuccess) { lbm_destroy(h); return fail(LBM_ERR_CUDA, "plan32: %s", cudaGetErrorString(e)); }
    }
    if (p->storage != LBM_F32 && !h->aa && 14 * h->plane < ((int64_t)1 << 31)) {
        h->s16.c = h->cf;
        for (int i = 0; i < 2; ++i) {
            h->s16.f[i] = h->buf[i];
            h->s16.g[i] = (float*)((char*)h->buf[i] + 9 * h->plane * f_size(p->storage));
        }
        h->s16.plane = h->plane;
        h->step16 = true;
    }
    // uniform porosity eps_mean, then the cold start
    const int thr = 256;
    const unsigned blocks = (unsigned)((h->N + thr - 1) / thr);
    DISPATCH_STO(p->storage, k_phi_fill<S_><<<blocks, thr, 0, h->stream>>>((PP<S_>*)h->phi, h->N, (float)p->eps_mean));
    e = cudaGetLastError();
    if (e == cudaSuccess) {
        rc = launch_init(h, nullptr, nullptr, nullptr);
        if (rc) { lbm_destroy(h); return rc; }
        e = cudaStreamSynchronize(h->stream);
    }
    if (e != cudaSuccess) {
        lbm_destroy(h);
        return fail(LBM_ERR_CUDA, "initialisation: %s", cudaGetErrorString(e));
    }
    *out = h;
    return LBM_OK;
}

int lbm_set_stream(lbm_handle* h, void* stream) {
    if (!h) return fail(LBM_ERR_INVALID, "handle is NULL");
    const cudaStream_t s = (cudaStream_t)stream;
    if (s == h->stream) return LBM_OK;
    CK(cudaSetDevice(h->device));
    // the new stream starts after everything already queued on the old one
    cudaEvent_t e = nullptr;
    CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    cudaError_t err = cudaEventRecord(e, h->stream);
    if (err == cudaSuccess) err = cudaStreamWaitEvent(s, e, 0);
    cudaEventDestroy(e);   // released once the recorded work has completed
    if (err != cudaSuccess) return fail(LBM_ERR_CUDA, "lbm_set_stream: %s", cudaGetErrorString(err));
    h->stream = s;
    return LBM_OK;
}

static int ensure_fstage(lbm_handle* h) {
    if (!h->fstage) CK(cudaMalloc((void**)&h->fstage, 3 * h->plane * sizeof(float)));
    return LBM_OK;
}

int lbm_set_porosity(lbm_handle* h, const float* phi, int on_device) {
    if (!h || !phi) return fail(LBM_ERR_INVALID, "NULL argument");
    CK(cudaSetDevice(h->device));
    if (int rc = wait_phi(h)) return rc;
    const float* src = phi;
    if (!on_device) {
        int rc = ensure_fstage(h);
        if (rc) return rc;
        CK(cudaMemcpyAsync(h->fstage, phi, h->N * sizeof(float), cudaMemcpyHostToDevice, h->stream));
        src = h->fstage;
    }
    CK(cudaMemsetAsync(h->bad, 0, sizeof(unsigned int), h->stream));
    DISPATCH_STO(h->p.storage, k_phi<S_><<<phi_blocks(h->N), 256, 0, h->stream>>>(src, (PP<S_>*)h->phi, h->N,
                                                                                   aligned16(src), h->bad));
    CK(cudaGetLastError());
    unsigned int bad = 0;
    CK(cudaMemcpyAsync(&bad, h->bad, sizeof(bad), cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    if (bad) return fail(LBM_ERR_INVALID, "%u porosity values outside (0, 1]", bad);
    return LBM_OK;
}

int lbm_set_porosity_async(lbm_handle* h, const float* phi) {
    if (!h || !phi) return fail(LBM_ERR_INVALID, "NULL argument");
    CK(cudaSetDevice(h->device));
    if (!h->copy_stream) {
        CK(cudaStreamCreateWithFlags(&h->copy_stream, cudaStreamNonBlocking));
        for (int i = 0; i < 2; ++i) {
            CK(cudaMalloc((void**)&h->astage[i], h->plane * sizeof(float)));   // may become the field
            CK(cudaEventCreateWithFlags(&h->consumed[i], cudaEventDisableTiming));
            CK(cudaEventCreateWithFlags(&h->copied[i], cudaEventDisableTiming));
        }
        CK(cudaMalloc((void**)&h->bad_async, sizeof(unsigned int)));
        CK(cudaMemsetAsync(h->bad_async, 0, sizeof(unsigned int), h->stream));
        CK(cudaStreamSynchronize(h->stream));
    }
    const int i = h->astage_i;
    h->astage_i ^= 1;
    // on the copy stream: staging buffer i is free once its last conversion has run, then
    // copy; the conversion into phi waits for the next reader of the field (wait_phi), so
    // copies follow one another on the copy stream while the compute stream runs, and an
    // upload that no reader saw is superseded by the next one
    CK(cudaStreamWaitEvent(h->copy_stream, h->consumed[i], 0));
    CK(cudaMemcpyAsync(h->astage[i], phi, h->N * sizeof(float), cudaMemcpyHostToDevice, h->copy_stream));
    CK(cudaEventRecord(h->copied[i], h->copy_stream));
    h->phi_pending = i;
    return LBM_OK;
}

int lbm_porosity_errors(lbm_handle* h, uint32_t* count, int clear) {
    if (!h || !count) return fail(LBM_ERR_INVALID, "NULL argument");
    *count = 0;
    if (!h->bad_async) return LBM_OK;
    CK(cudaSetDevice(h->device));
    int rc = wait_phi(h);
    if (rc) return rc;
    unsigned int v = 0;
    CK(cudaMemcpyAsync(&v, h->bad_async, sizeof(v), cudaMemcpyDeviceToHost, h->stream));
    if (clear) CK(cudaMemsetAsync(h->bad_async, 0, sizeof(unsigned int), h->stream));
    CK(cudaStreamSynchronize(h->stream));
    *count = v;
    return LBM_OK;
}

int lbm_init_fields(lbm_handle* h, const float* ur, const float* uz, const float* T, int on_device) {
    if (!h) return fail(LBM_ERR_INVALID, "handle is NULL");
    if ((ur == nullptr) != (uz == nullptr)) return fail(LBM_ERR_INVALID, "give both u_r and u_z or neither");
    CK(cudaSetDevice(h->device));
    const float *dur = ur, *duz = uz, *dT = T;
    if (!on_device && (ur || T)) {
        int rc = ensure_fstage(h);
        if (rc) return rc;
        if (ur) {
            CK(cudaMemcpyAsync(h->fstage, ur, h->N * sizeof(float), cudaMemcpyHostToDevice, h->stream));
            CK(cudaMemcpyAsync(h->fstage + h->plane, uz, h->N * sizeof(float), cudaMemcpyHostToDevice, h->stream));
            dur = h->fstage;
            duz = h->fstage + h->plane;
        }
        if (T) {
            CK(cudaMemcpyAsync(h->fstage + 2 * h->plane, T, h->N * sizeof(float), cudaMemcpyHostToDevice, h->stream));
            dT = h->fstage + 2 * h->plane;
        }
    }
    int rc = launch_init(h, dur, duz, dT);
    if (rc) return rc;
    if (!on_device) CK(cudaStreamSynchronize(h->stream));
    return LBM_OK;
}

// With 16-bit storage the flow reference is refreshed every LBM_FREF_EVERY steps of
// lbm_step (and before every check interval of lbm_run): the stored values stay of the
// size of the change since the last refresh however long the run.
constexpr int64_t LBM_FREF_EVERY = 1024;
static int launch_rebase(lbm_handle* h);

static int cur_lay(const lbm_handle* h) { return !h->aa ? LAY_N : (h->aa_odd ? LAY_L : LAY_S); }

// One step with in-place storage: read the current layout, write the other one, in the
// same buffer.  The wall kernel runs first: it reads the pre-collision values of its
// interior neighbours, which the bulk kernel overwrites.  One node per thread (update_column)
// for every storage type.
static int launch_step_inplace(lbm_handle* h, int nw) {
    cudaEvent_t e[4] = {nullptr, nullptr, nullptr, nullptr};   // wall start / end, bulk start / end
    if (h->timing)
        for (auto& x : e) CK(cudaEventCreate(&x));
    const bool i32 = 14 * h->plane < ((int64_t)1 << 31);
    const int64_t zblocks = (h->p.nz + BULK_THREADS - 1) / BULK_THREADS;
    const int rpt = (i32 && zblocks * ((h->p.nr + BULK_RPT - 1) / BULK_RPT) >= (int64_t)BULK_RPT_MIN_BLOCKS * h->sms) ? BULK_RPT : 1;
    const dim3 gb((unsigned)zblocks, (unsigned)((h->p.nr + rpt - 1) / rpt));
    const bool odd = h->aa_odd != 0;   // reading L (odd) or S (even)
    if (h->timing) CK(cudaEventRecord(e[0], h->stream));
#define AA_LAUNCH(LIN_, LOUT_)                                                                                  \
    DISPATCH_STO(h->p.storage, {                                                                               \
        const auto S = bufp<S_>(h, 0);                                                                         \
        const auto* ph = (const PP<S_>*)h->phi;                                                                \
        k_wall<S_, LIN_, LOUT_><<<(nw + 127) / 128, 128, 0, h->stream>>>(h->cf, S, S, ph, h->plane, nw);       \
        if (h->timing) CK(cudaEventRecord(e[1], h->stream));                                                   \
        if (h->timing) CK(cudaEventRecord(e[2], h->stream));                                                   \
        if (rpt > 1)                                                                                           \
            k_bulk<S_, int, BULK_RPT, LIN_, LOUT_><<<gb, BULK_THREADS, 0, h->stream>>>(h->cf, S, S, ph,         \
                                                                                        (int)h->plane);         \
        else if (i32)                                                                                          \
            k_bulk<S_, int, 1, LIN_, LOUT_><<<gb, BULK_THREADS, 0, h->stream>>>(h->cf, S, S, ph, (int)h->plane); \
        else                                                                                                   \
            k_bulk<S_, int64_t, 1, LIN_, LOUT_><<<gb, BULK_THREADS, 0, h->stream>>>(h->cf, S, S, ph, h->plane);  \
    })
    if (odd) {
        AA_LAUNCH(LAY_L, LAY_S);
    } else {
        AA_LAUNCH(LAY_S, LAY_L);
    }
#undef AA_LAUNCH
    CK(cudaGetLastError());
    if (h->timing) {
        CK(cudaEventRecord(e[3], h->stream));
        // the (bulk start, bulk end, wall start, wall end) quadruple lbm_kernel_times reads
        h->ev.push_back(e[2]);
        h->ev.push_back(e[3]);
        h->ev.push_back(e[0]);
        h->ev.push_back(e[1]);
    }
    h->aa_odd ^= 1;
    h->info.steps += 1;
    h->since_rebase += 1;
    return LBM_OK;
}

static int launch_step(lbm_handle* h) {
    if (int rc = wait_phi(h)) return rc;
    if (h->fref && h->since_rebase >= LBM_FREF_EVERY)
        if (int rc = launch_rebase(h)) return rc;
    const int nw = wall_count(h->p.geometry, h->p.nr, h->p.nz);
    if (h->aa) return launch_step_inplace(h, nw);
    // 16-bit storage: staged rows (below) for grids larger than STEP16_NODES with even nz, and where a
    // wait limit was set, since the staged kernel's waits are what the limit is for; else one launch
    // with the boundary nodes (FP16, per step: 2000 x 1500 49 against 59 us staged, 2000 x 2048 66
    // against 76, 2048 x 4096 129 either way, 4096 x 8192 504 against 455)
    constexpr int64_t STEP16_NODES = 8000000;
    const int64_t tiles16 = (int64_t)((h->p.nz + 2 * BULK_THREADS - 1) / (2 * BULK_THREADS)) * ((h->p.nr + BULK_RPT - 1) / BULK_RPT);
    const bool staged = h->stage && !(h->p.nz & 1) && tiles16 >= (int64_t)BULK_RPT_MIN_BLOCKS * h->sms &&
                        (h->N > STEP16_NODES || h->limit_set);
    if (h->step16 && !staged) {
        cudaEvent_t e[4] = {nullptr, nullptr, nullptr, nullptr};   // bulk start / end; no wall kernel
        if (h->timing) {
            CK(cudaEventCreate(&e[0]));
            CK(cudaEventCreate(&e[1]));
            CK(cudaEventRecord(e[0], h->stream));
        }
        h->s16.phi = (const float*)h->phi;
        CK(launch16(h->p.storage, h->s16, h->cur, h->stream));
        if (h->timing) {
            CK(cudaEventRecord(e[1], h->stream));
            for (auto x : e) h->ev.push_back(x);
        }
        h->cur ^= 1;
        h->info.steps += 1;
        h->since_rebase += 1;
        return LBM_OK;
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr, e1b = nullptr, e2 = nullptr;
    if (h->timing) {
        CK(cudaEventCreate(&e0));
        CK(cudaEventCreate(&e1));
        CK(cudaEventCreate(&e1b));
        CK(cudaEventCreate(&e2));
        CK(cudaEventRecord(e0, h->stream));
    }
    // BULK_RPT rows per thread where the grid keeps BULK_RPT_MIN_BLOCKS blocks per SM
    // (9 blocks of 128 threads are resident per SM), else one row per thread so that small
    // grids still fill the device
    const bool i32 = 14 * h->plane < ((int64_t)1 << 31);
    const int cols = staged ? 2 * BULK_THREADS : BULK_THREADS;
    const int64_t zblocks = (h->p.nz + cols - 1) / cols;
    const int rpt = (i32 && zblocks * ((h->p.nr + BULK_RPT - 1) / BULK_RPT) >= (int64_t)BULK_RPT_MIN_BLOCKS * h->sms) ? BULK_RPT : 1;
    const dim3 gb((unsigned)zblocks, (unsigned)((h->p.nr + rpt - 1) / rpt));
    if (h->step16) {
        DISPATCH_STO16(h->p.storage, {
            auto A = bufp<S_>(h, h->cur);
            auto B = bufp<S_>(h, h->cur ^ 1);
            const float* ph = (const float*)h->phi;
            if (h->p.nz % 8 == 0) k_bulk_stage<S_, BULK_RPT, true><<<gb, BULK_THREADS, 0, h->stream>>>(h->cf, A, B, ph, (int)h->plane, h->spin, h->wait_status);
            else k_bulk_stage<S_, BULK_RPT, false><<<gb, BULK_THREADS, 0, h->stream>>>(h->cf, A, B, ph, (int)h->plane, h->spin, h->wait_status);
        });
    } else if (i32) {   // FP32 storage with the discrete heater
        const auto k = rpt > 1 ? k_bulk<LBM_F32, int, BULK_RPT> : k_bulk<LBM_F32, int, 1>;
        k<<<gb, BULK_THREADS, 0, h->stream>>>(h->cf, bufp<LBM_F32>(h, h->cur), bufp<LBM_F32>(h, h->cur ^ 1),
                                              (const float*)h->phi, (int)h->plane);
    } else {
        DISPATCH_STO(h->p.storage,
                     k_bulk<S_, int64_t, 1><<<gb, BULK_THREADS, 0, h->stream>>>(
                         h->cf, bufp<S_>(h, h->cur), bufp<S_>(h, h->cur ^ 1), (const PP<S_>*)h->phi, h->plane));
    }
    CK(cudaGetLastError());
    if (h->timing) {
        CK(cudaEventRecord(e1, h->stream));
        CK(cudaEventRecord(e1b, h->stream));
    }
    // after the bulk kernel on the same stream (run beside it, the wall kernel took the
    // SMs the bulk kernel's memory pipeline needs: bulk 0.496 against 0.488 ms, FP16)
    DISPATCH_STO(h->p.storage,
                 k_wall<S_><<<(nw + 127) / 128, 128, 0, h->stream>>>(h->cf, bufp<S_>(h, h->cur), bufp<S_>(h, h->cur ^ 1),
                                                                     (const PP<S_>*)h->phi, h->plane, nw));
    CK(cudaGetLastError());
    if (h->timing) {
        CK(cudaEventRecord(e2, h->stream));
        // (bulk start, bulk end, wall start, wall end): the wall kernel starts where the bulk ends
        h->ev.push_back(e0);
        h->ev.push_back(e1);
        h->ev.push_back(e1b);
        h->ev.push_back(e2);
    }
    h->cur ^= 1;
    h->info.steps += 1;
    h->since_rebase += 1;
    return LBM_OK;
}

// n steps in one launch (lbm_f32.h), boundary nodes included.
static int launch_steps(lbm_handle* h, int n) {
    if (int rc = wait_phi(h)) return rc;
    cudaEvent_t e[4] = {nullptr, nullptr, nullptr, nullptr};   // bulk start / end; no wall kernel
    if (h->timing) {
        CK(cudaEventCreate(&e[0]));
        CK(cudaEventCreate(&e[1]));
        CK(cudaEventRecord(e[0], h->stream));
    }
    const auto state = [&](int which) {
        const Buf<LBM_F32> b = bufp<LBM_F32>(h, which);
        return State32{b.f, b.g};
    };
    CK(launch32(h->plan, h->c32, state(h->cur), state(h->cur ^ 1), (const float*)h->phi, (int)h->plane, n, h->stream));
    if (h->timing) {
        CK(cudaEventRecord(e[1], h->stream));
        for (auto x : e) h->ev.push_back(x);
    }
    h->cur ^= 1;
    h->info.steps += n;
    h->since_rebase += n;
    return LBM_OK;
}

int lbm_step(lbm_handle* h, int64_t nsteps) {
    if (!h) return fail(LBM_ERR_INVALID, "handle is NULL");
    if (nsteps < 0) return fail(LBM_ERR_INVALID, "nsteps < 0");
    CK(cudaSetDevice(h->device));
    const bool many = h->plan.two.strips != 0;
    // Launches alternate between the buffers.  A captured call is replayed on the buffers it was captured
    // with, so it takes an even number of launches for an even number of steps: where the plan would not,
    // its first launch is split.
    bool split = false;
    if (many && nsteps > 1) {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(h->stream, &cap) != cudaSuccess) (void)cudaGetLastError();
        split = cap == cudaStreamCaptureStatusActive && ((launches32(h->plan, nsteps) ^ nsteps) & 1);
    }
    int rest = 0;   // of a split launch
    for (int64_t s = 0; s < nsteps;) {
        int n = rest ? rest : many ? steps32(h->plan, nsteps - s) : 1;
        rest = 0;
        if (split) {
            rest = n - 1;
            n = 1;
            split = false;
        }
        const int rc = many ? launch_steps(h, n) : launch_step(h);
        if (rc) return rc;
        s += n;
    }
    return LBM_OK;
}

static int launch_moments(lbm_handle* h, int which, float* rho, float* ur, float* uz, float* T) {
    if (int rc = wait_phi(h)) return rc;
    if (h->plan.two.strips) {   // FP32 storage in two buffers (lbm_f32.h)
        const Buf<LBM_F32> b = bufp<LBM_F32>(h, which);
        CK(launch_fields32(h->c32, State32{b.f, b.g}, (const float*)h->phi, (int)h->plane, rho, ur, uz, T, h->stream));
        return LBM_OK;
    }
    if (h->step16) {            // 16-bit storage in two buffers (lbm_16.h)
        h->s16.phi = (const float*)h->phi;
        CK(launch_fields16(h->p.storage, h->s16, which, rho, ur, uz, T, h->stream));
        return LBM_OK;
    }
    const dim3 g = grid2d(h, 128);
    DISPATCH_LAY(cur_lay(h), DISPATCH_STO(h->p.storage,
                 k_moments<S_, L_><<<g, 128, 0, h->stream>>>(h->cf, bufp<S_>(h, which), (const PP<S_>*)h->phi,
                                                             h->plane, rho, ur, uz, T)));
    CK(cudaGetLastError());
    return LBM_OK;
}

static int ensure_mac(lbm_handle* h) {
    if (!h->mac) CK(cudaMalloc((void**)&h->mac, 8 * h->mstride * sizeof(float)));
    return LBM_OK;
}

int lbm_moments(lbm_handle* h, float* rho, float* ur, float* uz, float* T, int on_device) {
    if (!h) return fail(LBM_ERR_INVALID, "handle is NULL");
    CK(cudaSetDevice(h->device));
    if (on_device) return launch_moments(h, h->cur, rho, ur, uz, T);
    int rc = ensure_mac(h);
    if (rc) return rc;
    float* m = h->mac;
    rc = launch_moments(h, h->cur, m, m + h->mstride, m + 2 * h->mstride, m + 3 * h->mstride);
    if (rc) return rc;
    float* outs[4] = {rho, ur, uz, T};
    for (int j = 0; j < 4; ++j)
        if (outs[j])
            CK(cudaMemcpyAsync(outs[j], m + j * h->mstride, h->N * sizeof(float), cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    return LBM_OK;
}

// Eq. 42 of the current state into h->result[0..1] (stream-ordered).
static int launch_nusselt(lbm_handle* h) {
    const double dTw = h->p.T_hot - h->p.T_cold;
    const double ri = h->info.r0, ro = h->info.r0 + (h->p.nr - 1);
    const int blocks = (int)std::min<int64_t>((h->p.nz + 127) / 128, h->pblocks);
    DISPATCH_LAY(cur_lay(h), DISPATCH_STO(h->p.storage, k_nusselt<S_, L_><<<blocks, 128, 0, h->stream>>>(
                                                            h->cf, bufp<S_>(h, h->cur), h->plane, h->partials)));
    k_nusselt_final<<<1, 256, 0, h->stream>>>(h->partials, blocks, ri, ro, h->info.H, dTw, h->result);
    CK(cudaGetLastError());
    return LBM_OK;
}

int lbm_nusselt(lbm_handle* h, double* nu_inner, double* nu_outer) {
    if (!h) return fail(LBM_ERR_INVALID, "handle is NULL");
    if (h->p.geometry == LBM_PIPE_INFLOW || h->p.heater_len > 0) {   // lbm_pipe_nusselt, lbm_heater_nusselt
        if (nu_inner) *nu_inner = NAN;
        if (nu_outer) *nu_outer = NAN;
        return LBM_OK;
    }
    CK(cudaSetDevice(h->device));
    if (int rc = launch_nusselt(h)) return rc;
    double r[2];
    CK(cudaMemcpyAsync(r, h->result, sizeof(r), cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    if (nu_inner) *nu_inner = h->p.geometry == LBM_PIPE_PERIODIC_Z ? NAN : r[0];
    if (nu_outer) *nu_outer = r[1];
    return LBM_OK;
}

int lbm_nusselt_async(lbm_handle* h, double* out) {
    if (!h || !out) return fail(LBM_ERR_INVALID, "NULL argument");
    if (h->p.geometry == LBM_PIPE_INFLOW || h->p.heater_len > 0) {   // lbm_pipe_nusselt, lbm_heater_nusselt
        out[0] = out[1] = NAN;
        return LBM_OK;
    }
    CK(cudaSetDevice(h->device));
    if (int rc = launch_nusselt(h)) return rc;
    // stream order keeps h->result intact until it has been read
    const int pipe = h->p.geometry == LBM_PIPE_PERIODIC_Z;
    if (pipe) out[0] = NAN;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, out) == cudaSuccess && at.type == cudaMemoryTypeHost && at.devicePointer) {
        k_put2<<<1, 32, 0, h->stream>>>(h->result, (double*)at.devicePointer, pipe);
        CK(cudaGetLastError());
    } else {
        (void)cudaGetLastError();   // pageable memory: an ordinary copy
        CK(cudaMemcpyAsync(out + pipe, h->result + pipe, (2 - pipe) * sizeof(double), cudaMemcpyDeviceToHost,
                           h->stream));
    }
    return LBM_OK;
}

int lbm_sync(lbm_handle* h) {
    if (!h) return fail(LBM_ERR_INVALID, "handle is NULL");
    CK(cudaSetDevice(h->device));
    if (h->copy_stream) CK(cudaStreamSynchronize(h->copy_stream));
    CK(cudaStreamSynchronize(h->stream));
    return LBM_OK;
}

// FP64 residual sums between two field snapshots (4 planes each: rho, u_r, u_z, T):
// res = max(|du|_2 / |u|_2, |dT|_2 / |T|_2) over non-wall nodes, mass = sum r rho.
static int residual_between(lbm_handle* h, const float* cur, const float* prev, double* res, double* mass) {
    const int blocks = (int)std::min<int64_t>(h->pblocks, (h->N + 255) / 256);
    k_resid_partial<<<blocks, 256, 0, h->stream>>>(h->p.geometry, h->p.nr, h->p.nz, h->info.r0, cur, prev,
                                                   h->mstride, h->partials);
    CK(cudaGetLastError());
    k_sum_rows<<<1, 256, 0, h->stream>>>(h->partials, blocks, h->result);
    CK(cudaGetLastError());
    double s[RES_NV];
    CK(cudaMemcpyAsync(s, h->result, sizeof(s), cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    if (s[5] > 0) return fail(LBM_ERR_DIVERGED, "%.0f nodes hold NaN or Inf", s[5]);
    const double ru = s[1] > 0 ? std::sqrt(s[0] / s[1]) : (s[0] > 0 ? INFINITY : 0.0);
    const double rt = s[3] > 0 ? std::sqrt(s[2] / s[3]) : (s[2] > 0 ? INFINITY : 0.0);
    if (res) *res = ru > rt ? ru : rt;
    if (mass) *mass = s[4];
    return LBM_OK;
}

static int snapshot(lbm_handle* h, int which, float* m) {
    if (int rc = wait_phi(h)) return rc;
    return launch_moments(h, which, m, m + h->mstride, m + 2 * h->mstride, m + 3 * h->mstride);
}

int lbm_residual(lbm_handle* h, double* res, double* mass) {
    if (!h) return fail(LBM_ERR_INVALID, "handle is NULL");
    if (h->aa)
        return fail(LBM_ERR_INVALID, "in-place storage keeps no previous state: use lbm_run, or two snapshots and "
                                     "lbm_field_residual_noalloc");
    if (h->info.steps < 1) return fail(LBM_ERR_INVALID, "residual needs at least one step since initialisation");
    CK(cudaSetDevice(h->device));
    int rc = ensure_mac(h);
    if (rc) return rc;
    float* cur = h->mac;
    float* prev = h->mac + 4 * h->mstride;
    if ((rc = snapshot(h, h->cur, cur)) || (rc = snapshot(h, h->cur ^ 1, prev))) return rc;
    return residual_between(h, cur, prev, res, mass);
}

// Steady-state iteration.  The criterion is the mean change per step over each check
// interval, |u^n - u^(n-k)|_2 / (k |u^n|_2) (likewise T): with FP32 or 16-bit state the
// change between two consecutive steps carries rounding jitter of order 1e-8 - 1e-7
// that does not decay, whereas the interval mean falls with the true drift.
int lbm_run(lbm_handle* h, int64_t max_steps, int64_t check_every, double tol, int64_t* steps_done, double* res) {
    if (!h) return fail(LBM_ERR_INVALID, "handle is NULL");
    if (max_steps < 0 || check_every < 1) return fail(LBM_ERR_INVALID, "max_steps >= 0 and check_every >= 1 required");
    CK(cudaSetDevice(h->device));
    int rc = ensure_mac(h);
    if (rc) return rc;
    float* a = h->mac;
    float* b = h->mac + 4 * h->mstride;
    if ((rc = snapshot(h, h->cur, b))) return rc;
    int64_t done = 0;
    double r = INFINITY;
    while (done < max_steps) {
        const int64_t k = std::min(check_every, max_steps - done);
        if ((rc = lbm_rebase(h))) break;
        if ((rc = lbm_step(h, k))) break;
        done += k;
        if ((rc = lbm_wait_status(h, 0))) break;   // before the residual reads a state the timeout left invalid
        if ((rc = snapshot(h, h->cur, a))) break;
        double m;
        rc = residual_between(h, a, b, &r, &m);
        if (rc) break;
        r /= (double)k;
        std::swap(a, b);
        if (r <= tol) break;
    }
    if (steps_done) *steps_done = done;
    if (res) *res = r;
    return rc;
}

int lbm_pipe_nusselt(lbm_handle* h, double* nu, int32_t nz) {
    if (!h || !nu) return fail(LBM_ERR_INVALID, "NULL argument");
    if (h->p.geometry != LBM_PIPE_INFLOW) return fail(LBM_ERR_INVALID, "lbm_pipe_nusselt needs LBM_PIPE_INFLOW");
    if (nz != h->p.nz) return fail(LBM_ERR_INVALID, "nz = %d, the grid has %d", nz, h->p.nz);
    CK(cudaSetDevice(h->device));
    int rc = ensure_mac(h);
    if (rc) return rc;
    if ((rc = snapshot(h, h->cur, h->mac))) return rc;
    double* d = nullptr;
    CK(cudaMallocAsync((void**)&d, (size_t)nz * sizeof(double), h->stream));
    k_pipe_nusselt<<<(unsigned)((nz + 127) / 128), 128, 0, h->stream>>>(h->p.nr, nz, h->info.r0, h->mac + 2 * h->mstride,
                                                                       h->mac + 3 * h->mstride, d);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(nu, d, (size_t)nz * sizeof(double), cudaMemcpyDeviceToHost, h->stream);
    cudaFreeAsync(d, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return fail(LBM_ERR_CUDA, "pipe Nusselt: %s", cudaGetErrorString(e));
    return LBM_OK;
}

int lbm_heater_nusselt(lbm_handle* h, double* nu_mean, double* nu_z) {
    if (!h || !nu_mean) return fail(LBM_ERR_INVALID, "NULL argument");
    if (!(h->p.heater_len > 0)) return fail(LBM_ERR_INVALID, "lbm_heater_nusselt needs heater_len > 0");
    CK(cudaSetDevice(h->device));
    int rc = ensure_mac(h);
    if (rc) return rc;
    if ((rc = snapshot(h, h->cur, h->mac))) return rc;
    const int nz = h->p.nz;
    double* d = nullptr;
    CK(cudaMallocAsync((void**)&d, (size_t)(nz + 1) * sizeof(double), h->stream));
    k_heater_nusselt<<<1, 256, 0, h->stream>>>(nz, h->cf.hz0, h->cf.hz1, h->cf.periodic, h->p.T_hot - h->p.T_cold,
                                               h->p.T_cold, h->mac + 3 * h->mstride, d + 1, d);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(nu_mean, d, sizeof(double), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess && nu_z)
        e = cudaMemcpyAsync(nu_z, d + 1, (size_t)nz * sizeof(double), cudaMemcpyDeviceToHost, h->stream);
    cudaFreeAsync(d, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return fail(LBM_ERR_CUDA, "heater Nusselt: %s", cudaGetErrorString(e));
    return LBM_OK;
}

int lbm_stream_function(lbm_handle* h, float* psi, int on_device, double* psi_max) {
    if (!h) return fail(LBM_ERR_INVALID, "handle is NULL");
    CK(cudaSetDevice(h->device));
    int rc = ensure_mac(h);
    if (rc) return rc;
    if ((rc = snapshot(h, h->cur, h->mac))) return rc;
    const int nz = h->p.nz;
    const unsigned blocks = (unsigned)((nz + 127) / 128);
    float* dst = (psi && on_device) ? psi : h->mac + 4 * h->mstride;
    const int from_axis = h->p.geometry == LBM_PIPE_PERIODIC_Z || h->p.geometry == LBM_PIPE_INFLOW;
    double* d = nullptr;
    CK(cudaMallocAsync((void**)&d, (size_t)blocks * sizeof(double), h->stream));
    std::vector<double> bm(blocks);
    k_stream_function<<<blocks, 128, 0, h->stream>>>(h->p.nr, nz, h->info.r0, from_axis, h->mac + 2 * h->mstride,
                                                     dst, d);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(bm.data(), d, (size_t)blocks * sizeof(double), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess && psi && !on_device)
        e = cudaMemcpyAsync(psi, dst, (size_t)h->N * sizeof(float), cudaMemcpyDeviceToHost, h->stream);
    cudaFreeAsync(d, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return fail(LBM_ERR_CUDA, "stream function: %s", cudaGetErrorString(e));
    double big = 0;
    for (double x : bm) big = std::max(big, x);
    if (psi_max) *psi_max = big;
    return LBM_OK;
}

// Refresh the references of the current state: the temperature reference R(x) with FP32
// storage, the reference word (A, J, R) with 16-bit storage.
static int launch_rebase(lbm_handle* h) {
    const unsigned blocks = (unsigned)std::min<int64_t>((h->N + 255) / 256, (int64_t)h->sms * 16);
    if (h->p.storage == LBM_F32) {
        DISPATCH_LAY(cur_lay(h), k_rebase<LBM_F32, L_><<<blocks, 256, 0, h->stream>>>(
                                     h->cf, bufp<LBM_F32>(h, h->cur), h->plane, h->N, h->tref));
    } else {
        DISPATCH_LAY(cur_lay(h), DISPATCH_STO16(h->p.storage, k_rebase_16<S_, L_><<<blocks, 256, 0, h->stream>>>(
                                                                  h->cf, bufp<S_>(h, h->cur), h->plane, h->N, h->fref)));
    }
    CK(cudaGetLastError());
    h->since_rebase = 0;
    return LBM_OK;
}

int lbm_rebase(lbm_handle* h) {
    if (!h) return fail(LBM_ERR_INVALID, "handle is NULL");
    CK(cudaSetDevice(h->device));
    return launch_rebase(h);
}

int lbm_node_class(lbm_handle* h, uint8_t* out) {
    if (!h || !out) return fail(LBM_ERR_INVALID, "NULL argument");
    CK(cudaSetDevice(h->device));
    if (!h->cls) CK(cudaMalloc((void**)&h->cls, h->N));
    k_node_class<<<grid2d(h, 128), 128, 0, h->stream>>>(h->p.geometry, h->p.nr, h->p.nz, h->cls);
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(out, h->cls, h->N, cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    return LBM_OK;
}

int lbm_export_populations(lbm_handle* h, int32_t row0, int32_t nrows, double* f, double* g) {
    if (!h || !f || !g) return fail(LBM_ERR_INVALID, "NULL argument");
    if (row0 < 0 || nrows < 1 || row0 + nrows > h->p.nr) return fail(LBM_ERR_INVALID, "row range outside the grid");
    CK(cudaSetDevice(h->device));
    const int64_t P = (int64_t)nrows * h->p.nz;
    double* d = nullptr;
    CK(cudaMallocAsync((void**)&d, 14 * P * sizeof(double), h->stream));
    dim3 grid((unsigned)((h->p.nz + 127) / 128), (unsigned)nrows);
    DISPATCH_LAY(cur_lay(h), DISPATCH_STO(h->p.storage, k_export<S_, L_><<<grid, 128, 0, h->stream>>>(
                                                            h->cf, bufp<S_>(h, h->cur), h->plane, row0, nrows,
                                                            h->info.r0, h->info.T0, d)));
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(f, d, 9 * P * sizeof(double), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(g, d + 9 * P, 5 * P * sizeof(double), cudaMemcpyDeviceToHost, h->stream);
    cudaFreeAsync(d, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return fail(LBM_ERR_CUDA, "export: %s", cudaGetErrorString(e));
    return LBM_OK;
}

int lbm_get_info(lbm_handle* h, lbm_info* out) {
    if (!h || !out) return fail(LBM_ERR_INVALID, "NULL argument");
    *out = h->info;
    return LBM_OK;
}

int lbm_set_staging(lbm_handle* h, int enable) {
    if (!h) return fail(LBM_ERR_INVALID, "handle is NULL");
    h->stage = enable != 0;
    return LBM_OK;
}

int lbm_set_wait_limit(lbm_handle* h, int rounds) {
    if (!h) return fail(LBM_ERR_INVALID, "handle is NULL");
    h->spin = rounds < 0 ? STAGE_SPIN : rounds;
    h->limit_set = rounds >= 0;
    return LBM_OK;
}

int lbm_wait_status(lbm_handle* h, int clear) {
    if (!h) return fail(LBM_ERR_INVALID, "handle is NULL");
    if (!h->wait_status) return LBM_OK;
    CK(cudaSetDevice(h->device));
    int v = 0;
    CK(cudaMemcpyAsync(&v, h->wait_status, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    if (clear && v) CK(cudaMemsetAsync(h->wait_status, 0, sizeof(int), h->stream));
    if (v == LBM_ERR_TIMEOUT)
        return fail(LBM_ERR_TIMEOUT, "a bounded wait of the staged bulk kernel ran out (step results are invalid)");
    if (v) return fail(v, "the staged bulk kernel was launched for an odd nz (step results are invalid)");
    return LBM_OK;
}

int lbm_set_timing(lbm_handle* h, int enable) {
    if (!h) return fail(LBM_ERR_INVALID, "handle is NULL");
    CK(cudaSetDevice(h->device));
    CK(cudaStreamSynchronize(h->stream));
    for (auto e : h->ev)
        if (e) cudaEventDestroy(e);
    h->ev.clear();
    h->timing = enable != 0;
    return LBM_OK;
}

int lbm_kernel_times(lbm_handle* h, double* bulk_ms, int64_t* bulk_launches, double* wall_ms,
                     int64_t* wall_launches) {
    if (!h) return fail(LBM_ERR_INVALID, "handle is NULL");
    CK(cudaSetDevice(h->device));
    CK(cudaStreamSynchronize(h->stream));
    double tb = 0, tw = 0;
    int64_t nb = 0, nw = 0;
    for (size_t i = 0; i + 3 < h->ev.size(); i += 4) {   // (bulk start, bulk end, wall start, wall end)
        float a = 0, b = 0;
        CK(cudaEventElapsedTime(&a, h->ev[i], h->ev[i + 1]));
        tb += a;
        nb += 1;
        if (!h->ev[i + 2]) continue;   // a launch of several steps holds its boundary nodes
        CK(cudaEventElapsedTime(&b, h->ev[i + 2], h->ev[i + 3]));
        tw += b;
        nw += 1;
    }
    if (bulk_ms) *bulk_ms = tb;
    if (bulk_launches) *bulk_launches = nb;
    if (wall_ms) *wall_ms = tw;
    if (wall_launches) *wall_launches = nw;
    return LBM_OK;
}

const char* lbm_last_error(void) { return g_err.c_str(); }

}  // extern "C"

// ----------------------------------------------- allocation-free residual --
// Scratch for lbm_field_residual_noalloc: LBM_NOALLOC_ROWS partial rows of RES_NV
// doubles (one per reduction block) and one result row, 49 KB in total.  Every GPU
// that loads this library holds the array until the process exits.  Host code only
// ever passes the address obtained from cudaGetSymbolAddress; the symbol itself is a
// host-side stand-in there.
constexpr int LBM_NOALLOC_ROWS = 1024;
static __device__ __align__(256) double g_noalloc_scratch[(LBM_NOALLOC_ROWS + 1) * RES_NV];

// cuMemGetAddressRange of the driver, reached through the runtime's entry-point query so
// that the library does not link libcuda itself; NULL when the driver does not offer it.
typedef CUresult (*addr_range_fn)(CUdeviceptr* base, size_t* size, CUdeviceptr ptr);
static addr_range_fn addr_range() {
    static std::once_flag once;
    static addr_range_fn fn = nullptr;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (addr_range_fn)f;
        (void)cudaGetLastError();
    });
    return fn;
}

// A field-snapshot pointer must be device (or managed) memory of the current device
// whose allocation holds `bytes` from ptr on; checked without allocating anything.
static int check_field_ptr(const char* name, const float* ptr, int dev, size_t bytes) {
    cudaPointerAttributes at;
    const cudaError_t e = cudaPointerGetAttributes(&at, ptr);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return fail(LBM_ERR_INVALID, "%s: not a CUDA pointer (%s)", name, cudaGetErrorString(e));
    }
    if (at.type != cudaMemoryTypeDevice && at.type != cudaMemoryTypeManaged)
        return fail(LBM_ERR_INVALID, "%s: host or unregistered memory; device memory required", name);
    if (at.type == cudaMemoryTypeDevice && at.device != dev)
        return fail(LBM_ERR_INVALID, "%s: memory of device %d, current device %d", name, at.device, dev);
    if (addr_range_fn fn = addr_range()) {
        CUdeviceptr base = 0;
        size_t size = 0;
        if (fn(&base, &size, (CUdeviceptr)(uintptr_t)ptr) != CUDA_SUCCESS)
            return fail(LBM_ERR_INVALID, "%s: address range of the allocation unavailable", name);
        if ((uintptr_t)ptr + bytes > (uintptr_t)base + size)
            return fail(LBM_ERR_INVALID, "%s: its allocation ends %zu bytes after it, %zu needed", name,
                        (size_t)((uintptr_t)base + size - (uintptr_t)ptr), bytes);
    }
    return LBM_OK;
}

extern "C" int lbm_field_residual_noalloc(int32_t geometry, int32_t nr, int32_t nz, double r0, const float* cur,
                                          const float* prev, int64_t field_stride, double* res, double* mass,
                                          void* stream) {
    if (!cur || !prev || !res || !mass) return fail(LBM_ERR_INVALID, "NULL argument");
    if (geometry < 0 || geometry > 3) return fail(LBM_ERR_INVALID, "unknown geometry %d", geometry);
    if (nr < 3 || nz < 3 || nr > 65535 || nz > 65535 || (int64_t)nr * nz >= ((int64_t)1 << 31))
        return fail(LBM_ERR_INVALID, "grid %d x %d outside 3..65535 per side with nr*nz < 2^31", nr, nz);
    const int64_t N = (int64_t)nr * nz;
    if (field_stride < N || field_stride > ((int64_t)1 << 40))
        return fail(LBM_ERR_INVALID, "field_stride %lld outside [nr*nz, 2^40]", (long long)field_stride);
    int dev = 0;
    CK(cudaGetDevice(&dev));
    // both snapshots are read over their four planes: 3 * field_stride + nr * nz floats
    const size_t need = (size_t)(3 * field_stride + N) * sizeof(float);
    if (int rc = check_field_ptr("cur", cur, dev, need)) return rc;
    if (int rc = check_field_ptr("prev", prev, dev, need)) return rc;
    // the array's address in the current device's context, looked up on every call (a
    // lookup allocates nothing; an address kept from an earlier context could be stale)
    double* scratch = nullptr;
    CK(cudaGetSymbolAddress((void**)&scratch, g_noalloc_scratch));
    cudaStream_t s = (cudaStream_t)stream;
    const int blocks = (int)std::min<int64_t>(LBM_NOALLOC_ROWS, (N + 255) / 256);
    double* result = scratch + LBM_NOALLOC_ROWS * RES_NV;
    // every partial row the final sum reads is written by this call: nothing to clear
    k_resid_partial<<<blocks, 256, 0, s>>>(geometry, nr, nz, r0, cur, prev, field_stride, scratch);
    CK(cudaGetLastError());
    k_sum_rows<<<1, 256, 0, s>>>(scratch, blocks, result);
    CK(cudaGetLastError());
    double sum[RES_NV];
    CK(cudaMemcpyAsync(sum, result, sizeof(sum), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (sum[5] > 0) return fail(LBM_ERR_DIVERGED, "%.0f nodes hold NaN or Inf", sum[5]);
    const double ru = sum[1] > 0 ? std::sqrt(sum[0] / sum[1]) : (sum[0] > 0 ? INFINITY : 0.0);
    const double rt = sum[3] > 0 ? std::sqrt(sum[2] / sum[3]) : (sum[2] > 0 ? INFINITY : 0.0);
    *res = ru > rt ? ru : rt;
    *mass = sum[4];
    return LBM_OK;
}

// ======================================================================= batch ==
// Many independent problems of uneven size advanced by the same launches.
//
// Layout: one pooled device allocation holds, per instance, state A, state B and the
// porosity plane (each instance's own nr*nz, plane stride padded to 64 elements), and
// a second pool holds two field snapshots (4 planes each) per instance.  A device
// table of InstDesc carries each instance's lattice constants and pool offsets.
// A step is one launch covering every active instance (k_batch_step, lbm_f32.cu; k_batch_step16,
// lbm_16.cu; a second one if instances of both nz parities are present), or, for 16-bit batches
// above BATCH_STEP16_NODES or with a wait limit and FP32 batches with a discrete heater,
// k_batch_stage and k_batch_bulk over flattened lists of tiles (instance, first row, first column;
// k_batch_bulk's block shape chosen by lbm_batch_tune) beside k_batch_wall over the concatenated
// wall-node lists.  lbm_batch_run
// captures check_every steps (an even number, so every instance's A/B parity is the
// same at each check) in a CUDA graph and replays it; instances that reach the
// steady criterion leave the tile lists at the next check.
struct InstDesc {
    Consts<float> c;
    int64_t off_state[2];   // byte offsets of state buffers A and B in the state pool
    int64_t off_phi;        // byte offset of the porosity plane
    int64_t off_tref;       // byte offset of the reference-offset plane R(x) (FP16)
    int64_t off_fref;       // byte offset of the flow-reference plane Q(x) (16-bit storage)
    int64_t off_mac;        // float offset of the two field snapshots in the snapshot pool
    int64_t plane;          // elements per plane
    double r0, H, dTw;
};

template <int STO>
__device__ __forceinline__ Buf<STO> inst_buf(const InstDesc& d, char* pool, int which) {
    Buf<STO> b;
    b.f = (typename St<STO>::TF*)(pool + d.off_state[which]);
    b.g = (typename St<STO>::TG*)(pool + d.off_state[which] + 9 * d.plane * (int64_t)sizeof(typename St<STO>::TF));
    return b;
}

// Tile = (instance, first row, first column); block = (bz, rows); each thread updates
// RPT consecutive rows of its column (the instance descriptor is read once per thread).
// The per-node source is the single-problem kernel's (update_column); the two kernels
// agree to rounding (the compiler may fuse multiply-adds differently in each).
// Columns a thread of the bulk kernels covers: two with 16-bit storage (update_pair),
// one with FP32 storage.
template <int STO> __host__ __device__ constexpr int bulk_cols() { return has_fref<STO>() ? 2 : 1; }

#ifndef LBM_BATCH_DESC_SMEM
#define LBM_BATCH_DESC_SMEM 1
#endif
// 16-bit storage: the tiles of odd-nz instances (batch_rebuild orders them last), whose rows start at
// alternating alignment, so the pair update takes single loads.
template <int STO, int RPT>
__global__ void __launch_bounds__(256) k_batch_bulk(const InstDesc* __restrict__ desc, char* __restrict__ pool,
                                                    int parity, const int4* __restrict__ tiles) {
    const int4 t = tiles[blockIdx.x];
#if LBM_BATCH_DESC_SMEM
    // every thread of a tile works on the same instance: its descriptor in shared memory,
    // read from there where the per-node code needs a constant (no register copy of it)
    __shared__ InstDesc sd;
    {
        const int tid = threadIdx.y * blockDim.x + threadIdx.x;
        const int nw = (int)(sizeof(InstDesc) / sizeof(int));
        for (int w = tid; w < nw; w += blockDim.x * blockDim.y)
            reinterpret_cast<int*>(&sd)[w] = reinterpret_cast<const int*>(desc + t.x)[w];
        __syncthreads();
    }
    const InstDesc& d = sd;
    const Consts<float>& c = sd.c;
#else
    const InstDesc& d = desc[t.x];
    const Consts<float> c = d.c;
#endif
    const int kz = t.z + bulk_cols<STO>() * threadIdx.x;
    if (kz >= c.nz) return;
    const Buf<STO> A = inst_buf<STO>(d, pool, parity), B = inst_buf<STO>(d, pool, parity ^ 1);
    const typename St<STO>::P* phi = (const typename St<STO>::P*)(pool + d.off_phi);
    const int plane = (int)d.plane;
    if constexpr (has_fref<STO>()) {
        update_pair<STO, false>(c, A, B, phi, plane, t.y + threadIdx.y * RPT, RPT, kz);
    } else {
        update_column<STO, int>(c, A, B, phi, plane, t.y + threadIdx.y * RPT, RPT, kz);
    }
}

// 16-bit batches: the staged block (stage_block) over tiles (instance, first row, first
// column, rows) of BATCH_STAGE_NT column pairs of every active instance with even nz; the
// rows per tile (batch_stage_rows) are the same for all tiles of a batch.  On the sweep of 256 instances with Nr 64..512, 128-thread blocks at five
// per SM (the instance's pointers stay live: 102 registers allowed) measured 0.874 ms per
// step, 64-thread blocks 0.927 (ten per SM) and 0.969 (twelve, with spills), although
// 128-column tiles leave fewer thread slots idle on short rows (9 % against 17 %).
#ifndef LBM_BATCH_STAGE_NT
#define LBM_BATCH_STAGE_NT 128
#endif
#ifndef LBM_BATCH_STAGE_MIN_BLOCKS
#define LBM_BATCH_STAGE_MIN_BLOCKS 5
#endif
#ifndef LBM_BATCH_STAGE_MAX_ROWS
#define LBM_BATCH_STAGE_MAX_ROWS 16
#endif
constexpr int BATCH_STAGE_NT = LBM_BATCH_STAGE_NT;
template <int STO>
__global__ void __launch_bounds__(BATCH_STAGE_NT, LBM_BATCH_STAGE_MIN_BLOCKS) k_batch_stage(
    const InstDesc* __restrict__ desc, char* __restrict__ pool, int parity, const int4* __restrict__ tiles, int spin,
    int* __restrict__ status) {
    __shared__ PairStage<BATCH_STAGE_NT> sb;
    __shared__ InstDesc sd;   // the tile's instance: constants read from shared memory
    const int4 t = tiles[blockIdx.x];
    for (int w = threadIdx.x; w < (int)(sizeof(InstDesc) / sizeof(int)); w += BATCH_STAGE_NT)
        reinterpret_cast<int*>(&sd)[w] = reinterpret_cast<const int*>(desc + t.x)[w];
    __syncthreads();
    const Buf<STO> A = inst_buf<STO>(sd, pool, parity), B = inst_buf<STO>(sd, pool, parity ^ 1);
    stage_block<STO, BATCH_STAGE_NT, false>(sd.c, A, B, (const float*)(pool + sd.off_phi), (int)sd.plane, t.y, t.w, t.z,
                                            spin, status, sb);
}

// Flow reference refresh of every node the tiles cover (all nodes of the active instances),
// with the bulk kernels' tiles and block shape.
template <int STO, int RPT>
__global__ void __launch_bounds__(256) k_batch_rebase_flow(const InstDesc* __restrict__ desc, char* __restrict__ pool,
                                                           int parity, const int4* __restrict__ tiles) {
    if constexpr (has_fref<STO>()) {
        const int4 t = tiles[blockIdx.x];
        const InstDesc& d = desc[t.x];
        const Consts<float> c = d.c;
        const Buf<STO> S = inst_buf<STO>(d, pool, parity);
        uint2* fref = (uint2*)(pool + d.off_fref);
#pragma unroll 1
        for (int q = 0; q < RPT * bulk_cols<STO>(); ++q) {
            const int kr = t.y + threadIdx.y * RPT + q / bulk_cols<STO>();
            const int kz = t.z + bulk_cols<STO>() * threadIdx.x + q % bulk_cols<STO>();
            if (kr >= c.nr) break;
            if (kz >= c.nz) continue;
            rebase_16_node<STO, LAY_N, int>(c, S, (int)d.plane, kr, kz, kr * c.nz + kz, fref);
        }
    }
}

// Wall nodes of all active instances: prefix[k] = first wall thread of active instance k.
__device__ __forceinline__ int find_slot(const int* __restrict__ prefix, int n, int t) {
    int lo = 0, hi = n;   // prefix[lo] <= t < prefix[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (prefix[mid] <= t) lo = mid;
        else hi = mid;
    }
    return lo;
}

template <int STO>
__global__ void k_batch_wall(const InstDesc* __restrict__ desc, char* __restrict__ pool, int parity,
                             const int* __restrict__ active, const int* __restrict__ prefix, int nactive) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= prefix[nactive]) return;
    const int k = find_slot(prefix, nactive, t);
    const InstDesc& d = desc[active[k]];
    const Consts<float> c = d.c;
    int kr, kz;
    wall_node(c.geometry, c.nr, c.nz, t - prefix[k], kr, kz);
    const int cls = node_class(c.geometry, c.nr, c.nz, kr, kz);
    const Buf<STO> A = inst_buf<STO>(d, pool, parity), B = inst_buf<STO>(d, pool, parity ^ 1);
    const typename St<STO>::P* phi = (const typename St<STO>::P*)(pool + d.off_phi);
    float fh[9], gh[5], m0, rho, urb, uzb, dTb, refb;
    wall_state<STO>(c, A, phi, d.plane, cls, kr, kz, fh, gh, m0, rho, urb, uzb, dTb, refb);
    const int64_t n = (int64_t)kr * c.nz + kz;
    const float r = c.r0 + float(kr), ph = ldv(phi + n);
    float lin, nl, iph;
    porous(c, ph, lin, nl, iph);
    collide(c, r, rcp_acc(r), ph, lin, nl, iph, fh, gh, refb, m0, rho, urb, uzb, dTb);
    store<STO>(c, B, d.plane, kr, kz, n, fh, gh);
}

// Field snapshot `slot` (0 or 1) of every instance the tiles cover, all nodes.
template <int STO, int RPT>
__global__ void __launch_bounds__(256) k_batch_moments(const InstDesc* __restrict__ desc, char* __restrict__ pool,
                                                       float* __restrict__ macpool, int parity, int slot,
                                                       const int4* __restrict__ tiles) {
    const int4 t = tiles[blockIdx.x];
    const InstDesc& d = desc[t.x];
    const Consts<float> c = d.c;
    const Buf<STO> A = inst_buf<STO>(d, pool, parity);
    const typename St<STO>::P* phi = (const typename St<STO>::P*)(pool + d.off_phi);
    float* m = macpool + d.off_mac + (int64_t)slot * 4 * d.plane;
#pragma unroll 1
    for (int q = 0; q < RPT * bulk_cols<STO>(); ++q) {
        const int j = q / bulk_cols<STO>();
        const int kz = t.z + bulk_cols<STO>() * threadIdx.x + q % bulk_cols<STO>();
        const int kr = t.y + threadIdx.y * RPT + j;
        if (kr >= c.nr) break;
        if (kz >= c.nz) continue;
        const int cls = node_class(c.geometry, c.nr, c.nz, kr, kz);
        const int64_t n = (int64_t)kr * c.nz + kz;
        float fh[9], gh[5], m0, rho, ur = 0.f, uz = 0.f, dT, ref;
        if (is_wall(cls)) {
            wall_state<STO>(c, A, phi, d.plane, cls, kr, kz, fh, gh, m0, rho, ur, uz, dT, ref);
        } else {
            pull<STO>(c, A, d.plane, kr, kz, fh, gh, ref);
            const float r = c.r0 + float(kr), ph = ldv(phi + n);
            float lin, nl, iph;
            porous(c, ph, lin, nl, iph);
            recover(c, r, rcp_acc(r), ph, lin, nl, fh, gh, ref, m0, rho, ur, uz, dT);
        }
        m[n] = rho;
        m[d.plane + n] = ur;
        m[2 * d.plane + n] = uz;
        m[3 * d.plane + n] = (c.T0 + ref) + dT;
    }
}

// Per-instance residual sums between the two snapshots (cur = slot `cur`): grid
// (RB, nactive); partial rows [k][block][RES_NV].
constexpr int BATCH_RB = 16;
__global__ void k_batch_resid(const InstDesc* __restrict__ desc, const float* __restrict__ macpool, int cur,
                              const int* __restrict__ active, double* __restrict__ partials) {
    const int k = blockIdx.y;
    const InstDesc& d = desc[active[k]];
    const int nr = d.c.nr, nz = d.c.nz, geometry = d.c.geometry;
    const float* C = macpool + d.off_mac + (int64_t)cur * 4 * d.plane;
    const float* P = macpool + d.off_mac + (int64_t)(cur ^ 1) * 4 * d.plane;
    const int64_t fs = d.plane;
    double v[RES_NV] = {0, 0, 0, 0, 0, 0};
    const int64_t N = (int64_t)nr * nz;
    for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (int64_t)gridDim.x * blockDim.x) {
        const int kr = (int)(n / nz), kz = (int)(n - (int64_t)kr * nz);
        const float rho = C[n], ur = C[fs + n], uz = C[2 * fs + n], T = C[3 * fs + n];
        if (!isfinite(rho) || !isfinite(ur) || !isfinite(uz) || !isfinite(T)) v[5] += 1;
        v[4] += (d.r0 + kr) * (double)rho;
        if (is_wall(node_class(geometry, nr, nz, kr, kz))) continue;
        const double a = (double)ur - P[fs + n], b = (double)uz - P[2 * fs + n], e = (double)T - P[3 * fs + n];
        v[0] += a * a + b * b;
        v[1] += (double)ur * ur + (double)uz * uz;
        v[2] += e * e;
        v[3] += (double)T * T;
    }
    double out[RES_NV];
    block_sum<RES_NV>(v, out);
    if (threadIdx.x == 0)
        for (int j = 0; j < RES_NV; ++j) partials[((int64_t)k * gridDim.x + blockIdx.x) * RES_NV + j] = out[j];
}

__global__ void k_batch_resid_final(const double* __restrict__ partials, int rb, double* __restrict__ result) {
    const int k = blockIdx.x;
    double v[RES_NV] = {0, 0, 0, 0, 0, 0};
    for (int b = threadIdx.x; b < rb; b += blockDim.x)
        for (int j = 0; j < RES_NV; ++j) v[j] += partials[((int64_t)k * rb + b) * RES_NV + j];
    double out[RES_NV];
    block_sum<RES_NV>(v, out);
    if (threadIdx.x == 0)
        for (int j = 0; j < RES_NV; ++j) result[(int64_t)k * RES_NV + j] = out[j];
}

// Eq. 42 for every instance (one block each).
template <int STO>
__global__ void __launch_bounds__(256) k_batch_nusselt(const InstDesc* __restrict__ desc, char* __restrict__ pool,
                                                       const int* __restrict__ parity, double* __restrict__ result) {
    const InstDesc& d = desc[blockIdx.x];
    const Consts<float> c = d.c;
    const Buf<STO> A = inst_buf<STO>(d, pool, parity[blockIdx.x]);
    double v[2] = {0, 0};
    for (int kz = threadIdx.x; kz < c.nz; kz += blockDim.x) {
        const double wz = (kz == 0 || kz == c.nz - 1) ? 0.5 : 1.0;
        const double t0 = node_T<STO>(c, A, d.plane, 0, kz), t1 = node_T<STO>(c, A, d.plane, 1, kz);
        const double t2 = node_T<STO>(c, A, d.plane, 2, kz);
        const double u0 = node_T<STO>(c, A, d.plane, c.nr - 1, kz), u1 = node_T<STO>(c, A, d.plane, c.nr - 2, kz);
        const double u2 = node_T<STO>(c, A, d.plane, c.nr - 3, kz);
        v[0] += wz * (-3 * t0 + 4 * t1 - t2) * 0.5;
        v[1] += wz * (3 * u0 - 4 * u1 + u2) * 0.5;
    }
    double out[2];
    block_sum<2>(v, out);
    if (threadIdx.x == 0) {
        const double ro = d.r0 + (c.nr - 1);
        result[2 * blockIdx.x] = -d.r0 * out[0] / (d.H * d.dTw);
        result[2 * blockIdx.x + 1] = -ro * out[1] / (d.H * d.dTw);
    }
}

struct lbm_batch {
    int n = 0;
    int storage = 0;
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    // the wall kernel runs beside the bulk kernels on its own stream (fork / join per step)
    cudaStream_t wstream = nullptr;
    cudaEvent_t wfork = nullptr, wjoin = nullptr;
    std::vector<lbm_params> p;
    std::vector<lbm_info> info;
    std::vector<Consts<double>> cd;
    std::vector<InstDesc> desc;       // host copy
    InstDesc* d_desc = nullptr;
    char* pool = nullptr;
    float* macpool = nullptr;
    float* fstage = nullptr;          // largest instance: 3 planes (porosity or warm-start upload)
    int64_t max_plane = 0;
    int parity = 0;
    int64_t steps = 0;
    int64_t since_rebase = 0;         // steps since the last flow-reference refresh (16-bit)
    std::vector<char> active;         // 1 = still stepping
    // tiles and wall lists of the active set
    int bz = 128, rows = 1, rpt = 1;  // bulk block shape and rows per thread
    DeviceList tiles;                 // int4: active instances, all rows
    int ntiles = 0;
    int ntiles_even = 0;              // leading tiles of instances with even nz
    DeviceList act, prefix;           // int: active instances, their first wall threads
    int nactive = 0;
    int nwall = 0;
    double* partials = nullptr;
    double* result = nullptr;
    std::vector<int> iparity;         // buffer holding the state of an instance that stopped
    DeviceList stiles;                // int4, 16-bit: staged tiles of the active instances with even nz
    int nstiles = 0;
    int* wait_status = nullptr;       // 16-bit: LBM_ERR_TIMEOUT once a bounded wait of k_batch_stage ran out
    int spin = STAGE_SPIN;            // try_wait rounds of its per-row waits
    bool limit_set = false;           // by lbm_batch_set_wait_limit, to any value
    int stage = 1;                    // 16-bit: staged tiles for the even-nz instances (lbm_batch_set_staging)
    int sms = 0;                      // multiprocessors of the device
    // one launch per step (lbm_16.h)
    std::vector<Step16> inst16;
    std::vector<Inst32> inst32;
    Step16* d_inst16 = nullptr;
    DeviceList blocks16;              // int2, of the active instances: even nz, then odd nz
    int nblocks16[2] = {0, 0};
    bool step16 = false;              // it serves the active instances
    // one launch per step (lbm_f32.h), where it serves every instance
    bool step32 = false;
    Inst32* d_inst32 = nullptr;
    DeviceList blocks32;              // int2, of the active instances: even nz, then odd nz
    int nblocks32[2] = {0, 0};
    cudaGraphExec_t graph = nullptr;
    int64_t graph_steps = 0;
    int graph_parity = 0;             // batch parity the graph was captured at
    bool graph_dirty = true;
    int cur_parity(int i) const { return active[i] ? parity : iparity[i]; }
};

static void batch_free_graph(lbm_batch* b) {
    if (b->graph) cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
    b->graph_dirty = true;
}

// Rebuild the tile list, the active list and the wall prefix for the current active
// set and block shape.
// Rows per staged tile: the most (of 16, 8, 4, 2) that still leave the tiles at least four
// waves of resident blocks, since a block overlaps only the copies of its own next row
// with its compute (the 256-instance sweep ran at 0.844 ms per step with 16 rows, 0.847
// with 8, 0.874 with 4 and 0.944 with 2; 16 small instances of 1 M nodes at 31.8 us with
// 8 rows, 27.8 with 4 and 26.5 with 2).
static int batch_stage_rows(const lbm_batch* b, const std::vector<int>& act) {
    const int64_t want = 4LL * LBM_BATCH_STAGE_MIN_BLOCKS * b->sms;
    for (int r = LBM_BATCH_STAGE_MAX_ROWS; r > 2; r /= 2) {
        int64_t n = 0;
        for (int i : act)
            if (!(b->p[i].nz & 1))
                n += (int64_t)((b->p[i].nr + r - 1) / r) * ((b->p[i].nz + 2 * BATCH_STAGE_NT - 1) / (2 * BATCH_STAGE_NT));
        if (n >= want) return r;
    }
    return 2;
}

// 16-bit batches up to this many nodes take one launch per step from global loads (lbm_16.h), larger
// ones the staged tiles with the wall kernel beside them.  A batch whose wait limit was set runs
// staged: its waits are what the limit is for.
constexpr int64_t BATCH_STEP16_NODES = 8000000;
static int batch_rebuild(lbm_batch* b) {
    std::vector<int4> tiles, odd;   // tiles of instances with odd nz last (16-bit storage: k_batch_bulk's)
    std::vector<int> act, prefix(1, 0);
    for (int i = 0; i < b->n; ++i) {
        if (!b->active[i]) continue;
        act.push_back(i);
        prefix.push_back(prefix.back() + wall_count(b->p[i].geometry, b->p[i].nr, b->p[i].nz));
        const int zstep = b->bz * (b->storage == LBM_F32 ? 1 : 2);   // columns of a tile (bulk_cols)
        std::vector<int4>& dst = (b->p[i].nz & 1) ? odd : tiles;
        for (int kr = 0; kr < b->p[i].nr; kr += b->rows * b->rpt)
            for (int z0 = 0; z0 < b->p[i].nz; z0 += zstep) dst.push_back(make_int4(i, kr, z0, 0));
    }
    const int tiles_even = (int)tiles.size();
    tiles.insert(tiles.end(), odd.begin(), odd.end());
    std::vector<int4> st;
    if (b->storage != LBM_F32 && b->stage) {
        const int rpt = batch_stage_rows(b, act);
        for (int i : act)
            if (!(b->p[i].nz & 1))
                for (int kr = 0; kr < b->p[i].nr; kr += rpt)
                    for (int z0 = 0; z0 < b->p[i].nz; z0 += 2 * BATCH_STAGE_NT) st.push_back(make_int4(i, kr, z0, rpt));
    }
    int64_t nodes = 0;
    for (int i : act) nodes += (int64_t)b->p[i].nr * b->p[i].nz;
    const bool step16 = b->storage != LBM_F32 && (!b->stage || (nodes <= BATCH_STEP16_NODES && !b->limit_set));
    Blocks16 sb16;
    if (step16) sb16 = blocks16(b->p, act);
    StepBlocks sb32;
    if (b->step32) sb32 = blocks32(b->p, act);
    const int n16[2] = {(int)sb16.even.size(), (int)sb16.odd.size()}, n32[2] = {(int)sb32.even.size(), (int)sb32.odd.size()};
    sb16.even.insert(sb16.even.end(), sb16.odd.begin(), sb16.odd.end());
    sb32.even.insert(sb32.even.end(), sb32.odd.begin(), sb32.odd.end());
    const ListUpload lists[] = {{&b->tiles, tiles.data(), tiles.size() * sizeof(int4)},
                                {&b->stiles, st.data(), st.size() * sizeof(int4)},
                                {&b->blocks16, sb16.even.data(), sb16.even.size() * sizeof(int2)},
                                {&b->blocks32, sb32.even.data(), sb32.even.size() * sizeof(int2)},
                                {&b->act, act.data(), act.size() * sizeof(int)},
                                {&b->prefix, prefix.data(), prefix.size() * sizeof(int)}};
    CK(upload_lists(lists, 6, b->stream));
    // the counts follow the contents
    b->ntiles = (int)tiles.size();
    b->ntiles_even = tiles_even;
    b->nstiles = (int)st.size();
    b->step16 = step16;
    for (int k = 0; k < 2; ++k) {
        b->nblocks16[k] = n16[k];
        b->nblocks32[k] = n32[k];
    }
    b->nactive = (int)act.size();
    b->nwall = prefix.back();
    batch_free_graph(b);
    return LBM_OK;
}

// Another block shape; on an error the lists and the shape are as before.
static int batch_reshape(lbm_batch* b, int bz, int rows, int rpt) {
    const int old[3] = {b->bz, b->rows, b->rpt};
    b->bz = bz;
    b->rows = rows;
    b->rpt = rpt;
    const int rc = batch_rebuild(b);
    if (rc) {
        b->bz = old[0];
        b->rows = old[1];
        b->rpt = old[2];
    }
    return rc;
}

// Whether a step launches bulk tiles of that shape (k_batch_bulk).
static bool batch_bulk_tiles(const lbm_batch* b) {
    return !b->step32 && !b->step16 && (b->storage == LBM_F32 || b->ntiles > b->ntiles_even);
}

template <int STO> static Buf<STO> batch_buf(const lbm_batch* b, int i, int which) {
    const InstDesc& d = b->desc[i];
    Buf<STO> r;
    r.f = (typename St<STO>::TF*)(b->pool + d.off_state[which]);
    r.g = (typename St<STO>::TG*)(b->pool + d.off_state[which] + 9 * d.plane * (int64_t)sizeof(typename St<STO>::TF));
    return r;
}

// Flow-reference refresh of every active instance (16-bit storage), one launch.
static int batch_launch_rebase_flow(lbm_batch* b) {
    if (b->storage != LBM_F32 && b->nactive) {
        const dim3 blk(b->bz, b->rows);
        DISPATCH_STO16(b->storage, DISPATCH_RPT(b->rpt, k_batch_rebase_flow<S_, R_><<<b->ntiles, blk, 0, b->stream>>>(
                                                            b->d_desc, b->pool, b->parity, (const int4*)b->tiles.dev)));
        CK(cudaGetLastError());
    }
    b->since_rebase = 0;
    return LBM_OK;
}

static int batch_launch_step(lbm_batch* b) {
    if (!b->nactive) return LBM_OK;
    // 16-bit storage: the refresh of lbm_step, every LBM_FREF_EVERY steps since the last
    if (b->storage != LBM_F32 && b->since_rebase >= LBM_FREF_EVERY)
        if (int rc = batch_launch_rebase_flow(b)) return rc;
    if (b->step16) {
        for (int odd = 0; odd < 2; ++odd)
            if (b->nblocks16[odd])
                CK(launch_batch16(b->storage, b->d_inst16, (const int2*)b->blocks16.dev + (odd ? b->nblocks16[0] : 0), b->nblocks16[odd],
                                  odd != 0, b->parity, b->stream));
        b->parity ^= 1;
        b->since_rebase += 1;
        return LBM_OK;
    }
    if (b->step32) {
        for (int odd = 0; odd < 2; ++odd)
            if (b->nblocks32[odd])
                CK(launch_batch32(b->d_inst32, (const int2*)b->blocks32.dev + (odd ? b->nblocks32[0] : 0), b->nblocks32[odd], odd != 0,
                                  b->parity, b->stream));
        b->parity ^= 1;
        b->since_rebase += 1;
        return LBM_OK;
    }
    // the wall kernel reads only the pre-step states and writes only boundary nodes, which
    // the bulk kernels do not touch: it runs beside them on the wall stream
    CK(cudaEventRecord(b->wfork, b->stream));
    CK(cudaStreamWaitEvent(b->wstream, b->wfork, 0));
    DISPATCH_STO(b->storage, k_batch_wall<S_><<<(b->nwall + 127) / 128, 128, 0, b->wstream>>>(
                                 b->d_desc, b->pool, b->parity, (const int*)b->act.dev, (const int*)b->prefix.dev, b->nactive));
    CK(cudaGetLastError());
    const dim3 blk(b->bz, b->rows);
    if (b->storage == LBM_F32) {
        DISPATCH_RPT(b->rpt, k_batch_bulk<LBM_F32, R_><<<b->ntiles, blk, 0, b->stream>>>(
                                 b->d_desc, b->pool, b->parity, (const int4*)b->tiles.dev));
    } else {
        const int ne = b->ntiles_even, no = b->ntiles - b->ntiles_even;
        if (b->nstiles)   // even nz: staged tiles
            DISPATCH_STO16(b->storage, k_batch_stage<S_><<<b->nstiles, BATCH_STAGE_NT, 0, b->stream>>>(
                                           b->d_desc, b->pool, b->parity, (const int4*)b->stiles.dev, b->spin, b->wait_status));
        if (no)
            DISPATCH_STO16(b->storage, DISPATCH_RPT(b->rpt, k_batch_bulk<S_, R_><<<no, blk, 0, b->stream>>>(
                                                                b->d_desc, b->pool, b->parity, (const int4*)b->tiles.dev + ne)));
    }
    CK(cudaGetLastError());
    CK(cudaEventRecord(b->wjoin, b->wstream));
    CK(cudaStreamWaitEvent(b->stream, b->wjoin, 0));
    b->parity ^= 1;
    b->since_rebase += 1;
    return LBM_OK;
}

extern "C" {

int lbm_batch_destroy(lbm_batch* b) {
    if (!b) return LBM_OK;
    cudaSetDevice(b->device);
    if (b->stream) cudaStreamSynchronize(b->stream);
    if (b->wstream) {
        cudaStreamSynchronize(b->wstream);
        cudaStreamDestroy(b->wstream);
    }
    if (b->wfork) cudaEventDestroy(b->wfork);
    if (b->wjoin) cudaEventDestroy(b->wjoin);
    batch_free_graph(b);
    cudaFree(b->d_desc);
    cudaFree(b->pool);
    cudaFree(b->macpool);
    cudaFree(b->fstage);
    for (DeviceList* l : {&b->tiles, &b->stiles, &b->blocks16, &b->blocks32, &b->act, &b->prefix}) cudaFree(l->dev);
    cudaFree(b->d_inst32);
    cudaFree(b->d_inst16);
    cudaFree(b->wait_status);
    cudaFree(b->partials);
    cudaFree(b->result);
    if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
    delete b;
    return LBM_OK;
}

int lbm_batch_create(const lbm_params* p, int32_t n, lbm_batch** out) {
    if (!p || !out || n < 1) return fail(LBM_ERR_INVALID, "need params[n], n >= 1 and an output pointer");
    *out = nullptr;
    lbm_batch* b = new lbm_batch();
    b->n = n;
    b->storage = p[0].storage;
    b->p.assign(p, p + n);
    b->info.resize(n);
    b->cd.resize(n);
    b->desc.resize(n);
    int64_t state_off = 0, mac_off = 0;
    for (int i = 0; i < n; ++i) {
        int rc = derive(&p[i], &b->info[i], &b->cd[i]);
        if (rc) { delete b; return fail(rc, "instance %d: %s", i, g_err.c_str()); }
        if (p[i].storage != b->storage) { delete b; return fail(LBM_ERR_INVALID, "instance %d: storage differs", i); }
        if (p[i].inplace) { delete b; return fail(LBM_ERR_INVALID, "instance %d: in-place storage is for lbm_create", i); }
        const int64_t N = (int64_t)p[i].nr * p[i].nz, plane = (N + 63) / 64 * 64;
        if (14 * plane >= ((int64_t)1 << 31)) { delete b; return fail(LBM_ERR_INVALID, "instance %d too large", i); }
        InstDesc& d = b->desc[i];
        d.c = to_float(b->cd[i]);
        d.plane = plane;
        d.off_state[0] = state_off;
        state_off += (int64_t)state_bytes(b->storage, plane);
        d.off_state[1] = state_off;
        state_off += (int64_t)state_bytes(b->storage, plane);
        d.off_phi = state_off;
        state_off += (plane * (int64_t)phi_size(b->storage) + 255) / 256 * 256;
        d.off_tref = state_off;   // R(x) plane (FP32 storage) or reference words (16-bit storage)
        d.off_fref = state_off;
        state_off += (plane * (int64_t)(p[i].storage == LBM_F32 ? sizeof(__half) : sizeof(uint2)) + 255) / 256 * 256;
        d.off_mac = mac_off;
        mac_off += 8 * plane;
        d.r0 = b->info[i].r0;
        d.H = b->info[i].H;
        d.dTw = p[i].T_hot - p[i].T_cold;
        b->max_plane = std::max(b->max_plane, plane);
    }
    b->active.assign(n, 1);
    b->iparity.assign(n, 0);
    cudaError_t e = cudaGetDevice(&b->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, b->device);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&b->wstream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->wfork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->wjoin, cudaEventDisableTiming);
    b->own_stream = e == cudaSuccess;
    if (e == cudaSuccess) e = cudaMalloc((void**)&b->pool, state_off);
    if (e == cudaSuccess)
        for (int i = 0; i < n; ++i) {
            const __half* tr = b->storage == LBM_F32 ? (const __half*)(b->pool + b->desc[i].off_tref) : nullptr;
            b->desc[i].c.tref = tr;
            b->cd[i].tref = tr;
            const uint2* fr = b->storage == LBM_F32 ? nullptr : (const uint2*)(b->pool + b->desc[i].off_fref);
            b->desc[i].c.fref = fr;
            b->cd[i].fref = fr;
        }
    if (e == cudaSuccess) e = cudaMalloc((void**)&b->macpool, mac_off * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc((void**)&b->d_desc, n * sizeof(InstDesc));
    if (e == cudaSuccess) e = cudaMalloc((void**)&b->partials, (size_t)n * BATCH_RB * RES_NV * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void**)&b->result, (size_t)n * RES_NV * sizeof(double));
    if (e == cudaSuccess && b->storage != LBM_F32) {
        e = cudaMalloc((void**)&b->wait_status, sizeof(int));
        if (e == cudaSuccess) e = cudaMemsetAsync(b->wait_status, 0, sizeof(int), b->stream);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(b->storage == LBM_F16 ? k_batch_stage<LBM_F16> : k_batch_stage<LBM_BF16>,
                                     cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
    }
    if (e == cudaSuccess && b->storage != LBM_F32) {
        std::vector<Step16>& inst = b->inst16;
        inst.resize(n);
        for (int i = 0; i < n; ++i) {
            const InstDesc& d = b->desc[i];
            inst[i].c = d.c;
            for (int k = 0; k < 2; ++k) {
                inst[i].f[k] = b->pool + d.off_state[k];
                inst[i].g[k] = (float*)(b->pool + d.off_state[k] + 9 * d.plane * (int64_t)f_size(b->storage));
            }
            inst[i].phi = (const float*)(b->pool + d.off_phi);
            inst[i].plane = d.plane;
        }
        e = cudaMalloc((void**)&b->d_inst16, n * sizeof(Step16));
        if (e == cudaSuccess) e = cudaMemcpy(b->d_inst16, inst.data(), n * sizeof(Step16), cudaMemcpyHostToDevice);
    }
    b->step32 = true;
    for (int i = 0; i < n; ++i) b->step32 = b->step32 && serves32(p[i]);
    if (e == cudaSuccess && b->step32) {
        std::vector<Inst32>& inst = b->inst32;
        inst.resize(n);
        for (int i = 0; i < n; ++i) {
            inst[i].c = consts32(b->cd[i], b->desc[i].c);
            for (int k = 0; k < 2; ++k) {
                const Buf<LBM_F32> s = batch_buf<LBM_F32>(b, i, k);
                inst[i].s[k] = State32{s.f, s.g};
            }
            inst[i].phi = (const float*)(b->pool + b->desc[i].off_phi);
            inst[i].plane = (int)b->desc[i].plane;
        }
        e = cudaMalloc((void**)&b->d_inst32, n * sizeof(Inst32));
        if (e == cudaSuccess) e = cudaMemcpy(b->d_inst32, inst.data(), n * sizeof(Inst32), cudaMemcpyHostToDevice);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(b->d_desc, b->desc.data(), n * sizeof(InstDesc), cudaMemcpyHostToDevice,
                                              b->stream);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        lbm_batch_destroy(b);
        return fail(e == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA, "batch allocation: %s",
                    cudaGetErrorString(e));
    }
    // uniform porosity and the cold start of every instance
    for (int i = 0; i < n; ++i) {
        const InstDesc& d = b->desc[i];
        const int64_t N = (int64_t)p[i].nr * p[i].nz;
        const dim3 g((unsigned)((p[i].nz + 127) / 128), (unsigned)p[i].nr);
        DISPATCH_STO(b->storage, {
            k_phi_fill<S_><<<(unsigned)((N + 255) / 256), 256, 0, b->stream>>>((PP<S_>*)(b->pool + d.off_phi), N,
                                                                                (float)p[i].eps_mean);
            k_init<S_><<<g, 128, 0, b->stream>>>(b->cd[i], batch_buf<S_>(b, i, 0), (const PP<S_>*)(b->pool + d.off_phi),
                                                 d.plane, nullptr, nullptr, nullptr, p[i].init_noise, p[i].seed,
                                                 (__half*)(b->pool + d.off_tref), (uint2*)b->cd[i].fref, 0);
        });
    }
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) {
        lbm_batch_destroy(b);
        return fail(LBM_ERR_CUDA, "batch initialisation: %s", cudaGetErrorString(e));
    }
    int rc = batch_rebuild(b);
    if (rc) { lbm_batch_destroy(b); return rc; }
    *out = b;
    return LBM_OK;
}

int lbm_batch_set_stream(lbm_batch* b, void* stream) {
    if (!b) return fail(LBM_ERR_INVALID, "batch is NULL");
    if (!stream) return fail(LBM_ERR_INVALID, "a batch needs a created stream (graph capture)");
    CK(cudaSetDevice(b->device));
    CK(cudaStreamSynchronize(b->stream));
    if (b->own_stream) cudaStreamDestroy(b->stream);
    b->own_stream = false;
    b->stream = (cudaStream_t)stream;
    batch_free_graph(b);
    return LBM_OK;
}

static int batch_upload(lbm_batch* b, const float* src, int64_t N, int slot, const float** dev) {
    if (!b->fstage) CK(cudaMalloc((void**)&b->fstage, 3 * b->max_plane * sizeof(float)));
    CK(cudaMemcpyAsync(b->fstage + slot * b->max_plane, src, N * sizeof(float), cudaMemcpyHostToDevice, b->stream));
    *dev = b->fstage + slot * b->max_plane;
    return LBM_OK;
}

int lbm_batch_set_porosity(lbm_batch* b, int32_t i, const float* phi, int on_device) {
    if (!b || !phi || i < 0 || i >= b->n) return fail(LBM_ERR_INVALID, "bad batch, instance or pointer");
    CK(cudaSetDevice(b->device));
    const int64_t N = (int64_t)b->p[i].nr * b->p[i].nz;
    const float* src = phi;
    int rc;
    if (!on_device && (rc = batch_upload(b, phi, N, 0, &src))) return rc;
    unsigned int* bad = (unsigned int*)b->result;   // scratch word
    CK(cudaMemsetAsync(bad, 0, sizeof(unsigned int), b->stream));
    DISPATCH_STO(b->storage, k_phi<S_><<<phi_blocks(N), 256, 0, b->stream>>>(
                                 src, (PP<S_>*)(b->pool + b->desc[i].off_phi), N, aligned16(src), bad));
    CK(cudaGetLastError());
    unsigned int nb = 0;
    CK(cudaMemcpyAsync(&nb, bad, sizeof(nb), cudaMemcpyDeviceToHost, b->stream));
    CK(cudaStreamSynchronize(b->stream));
    if (nb) return fail(LBM_ERR_INVALID, "instance %d: %u porosity values outside (0, 1]", i, nb);
    return LBM_OK;
}

int lbm_batch_init_fields(lbm_batch* b, int32_t i, const float* ur, const float* uz, const float* T, int on_device) {
    if (!b || i < 0 || i >= b->n) return fail(LBM_ERR_INVALID, "bad batch or instance");
    if ((ur == nullptr) != (uz == nullptr)) return fail(LBM_ERR_INVALID, "give both u_r and u_z or neither");
    CK(cudaSetDevice(b->device));
    const int64_t N = (int64_t)b->p[i].nr * b->p[i].nz;
    const float *dur = ur, *duz = uz, *dT = T;
    int rc;
    if (!on_device) {
        if (ur && ((rc = batch_upload(b, ur, N, 0, &dur)) || (rc = batch_upload(b, uz, N, 1, &duz)))) return rc;
        if (T && (rc = batch_upload(b, T, N, 2, &dT))) return rc;
    }
    const InstDesc& d = b->desc[i];
    const dim3 g((unsigned)((b->p[i].nz + 127) / 128), (unsigned)b->p[i].nr);
    // the instance's current buffer is the batch parity
    DISPATCH_STO(b->storage, k_init<S_><<<g, 128, 0, b->stream>>>(b->cd[i], batch_buf<S_>(b, i, b->parity),
                                                                   (const PP<S_>*)(b->pool + d.off_phi), d.plane, dur,
                                                                   duz, dT, b->p[i].init_noise, b->p[i].seed,
                                                                   (__half*)(b->pool + d.off_tref), (uint2*)b->cd[i].fref,
                                                                   0));
    CK(cudaGetLastError());
    CK(cudaStreamSynchronize(b->stream));
    if (!b->active[i]) {
        b->active[i] = 1;
        const int rc = batch_rebuild(b);
        if (rc) b->active[i] = 0;   // the lists are as before
        return rc;
    }
    return LBM_OK;
}

int lbm_batch_step(lbm_batch* b, int64_t nsteps) {
    if (!b || nsteps < 0) return fail(LBM_ERR_INVALID, "bad batch or nsteps");
    CK(cudaSetDevice(b->device));
    for (int64_t s = 0; s < nsteps; ++s) {
        int rc = batch_launch_step(b);
        if (rc) return rc;
    }
    b->steps += nsteps;
    return LBM_OK;
}

// Reference refresh of instance i (the kernel of lbm_rebase, on the instance's current
// buffer).
static int batch_rebase_one(lbm_batch* b, int i) {
    const InstDesc& d = b->desc[i];
    const int64_t N = (int64_t)b->p[i].nr * b->p[i].nz;
    const unsigned blocks = (unsigned)std::min<int64_t>((N + 255) / 256, 4096);
    if (b->storage == LBM_F32) {
        k_rebase<LBM_F32><<<blocks, 256, 0, b->stream>>>(d.c, batch_buf<LBM_F32>(b, i, b->cur_parity(i)), d.plane, N,
                                                         (__half*)(b->pool + d.off_tref));
    } else {
        DISPATCH_STO16(b->storage, k_rebase_16<S_><<<blocks, 256, 0, b->stream>>>(
                                       d.c, batch_buf<S_>(b, i, b->cur_parity(i)), d.plane, N,
                                       (uint2*)(b->pool + d.off_fref)));
    }
    CK(cudaGetLastError());
    return LBM_OK;
}

int lbm_batch_rebase(lbm_batch* b) {
    if (!b) return fail(LBM_ERR_INVALID, "batch is NULL");
    CK(cudaSetDevice(b->device));
    for (int i = 0; i < b->n; ++i) {
        int rc = batch_rebase_one(b, i);
        if (rc) return rc;
    }
    b->since_rebase = 0;
    return LBM_OK;
}

// Snapshot `slot` of every active instance.
static int batch_snapshot(lbm_batch* b, int slot) {
    // moments use all rows of the active instances: the bulk tiles cover them
    const dim3 blk(b->bz, b->rows);
    DISPATCH_STO(b->storage, DISPATCH_RPT(b->rpt, k_batch_moments<S_, R_><<<b->ntiles, blk, 0, b->stream>>>(
                                                       b->d_desc, b->pool, b->macpool, b->parity, slot, (const int4*)b->tiles.dev)));
    CK(cudaGetLastError());
    return LBM_OK;
}

int lbm_batch_run(lbm_batch* b, int64_t max_steps, int64_t check_every, double tol, int64_t* steps_out,
                  double* res_out) {
    if (!b) return fail(LBM_ERR_INVALID, "batch is NULL");
    if (max_steps < 0 || check_every < 2 || (check_every & 1))
        return fail(LBM_ERR_INVALID, "max_steps >= 0 and an even check_every >= 2 required");
    CK(cudaSetDevice(b->device));
    std::vector<int64_t> done(b->n, 0);
    std::vector<double> res(b->n, INFINITY);
    int slot = 0;
    int rc = batch_snapshot(b, slot ^ 1);
    if (rc) return rc;
    int64_t total = 0;
    while (total < max_steps && b->nactive > 0) {
        const int64_t k = std::min(check_every, max_steps - total);
        // reference refresh before every check interval, as lbm_run does
        if (b->step32) {
            int64_t most = 0;
            for (int i = 0; i < b->n; ++i)
                if (b->active[i]) most = std::max(most, (int64_t)b->p[i].nr * b->p[i].nz);
            CK(launch_batch_rebase32(b->d_inst32, (const int*)b->act.dev, b->nactive, most, b->parity, b->stream));
        } else if (b->storage == LBM_F32) {
            for (int i = 0; i < b->n; ++i)
                if (b->active[i] && (rc = batch_rebase_one(b, i))) return rc;
        } else if ((rc = batch_launch_rebase_flow(b))) {
            return rc;
        }
        b->since_rebase = 0;
        if (k == check_every) {
            if (b->graph_dirty || b->graph_steps != k || b->graph_parity != b->parity) {
                batch_free_graph(b);
                cudaGraph_t g = nullptr;
                CK(cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal));
                const int p0 = b->parity;
                for (int64_t s = 0; s < k; ++s) {
                    rc = batch_launch_step(b);
                    if (rc) break;
                }
                b->parity = p0;   // replays start from the same parity (k is even)
                cudaError_t e = cudaStreamEndCapture(b->stream, &g);
                if (rc) { if (g) cudaGraphDestroy(g); return rc; }
                if (e != cudaSuccess) return fail(LBM_ERR_CUDA, "graph capture: %s", cudaGetErrorString(e));
                e = cudaGraphInstantiate(&b->graph, g, 0);
                cudaGraphDestroy(g);
                if (e != cudaSuccess) return fail(LBM_ERR_CUDA, "graph instantiate: %s", cudaGetErrorString(e));
                b->graph_steps = k;
                b->graph_parity = p0;
                b->graph_dirty = false;
            }
            CK(cudaGraphLaunch(b->graph, b->stream));
        } else {
            for (int64_t s = 0; s < k; ++s)
                if ((rc = batch_launch_step(b))) return rc;
            // an odd tail leaves the parity flipped, which the launches already track
        }
        total += k;
        b->steps += k;
        for (int i = 0; i < b->n; ++i)
            if (b->active[i]) done[i] += k;
        if ((rc = lbm_batch_wait_status(b, 0))) return rc;   // before the residual reads an invalid state
        if ((rc = batch_snapshot(b, slot))) return rc;
        const dim3 grid(BATCH_RB, b->nactive);
        k_batch_resid<<<grid, 256, 0, b->stream>>>(b->d_desc, b->macpool, slot, (const int*)b->act.dev, b->partials);
        CK(cudaGetLastError());
        k_batch_resid_final<<<b->nactive, 256, 0, b->stream>>>(b->partials, BATCH_RB, b->result);
        CK(cudaGetLastError());
        std::vector<double> s((size_t)b->nactive * RES_NV);
        CK(cudaMemcpyAsync(s.data(), b->result, s.size() * sizeof(double), cudaMemcpyDeviceToHost, b->stream));
        CK(cudaStreamSynchronize(b->stream));
        std::vector<int> act;
        for (int i = 0; i < b->n; ++i)
            if (b->active[i]) act.push_back(i);
        bool changed = false;
        const auto was_active = b->active;
        int diverged = -1;
        for (int j = 0; j < b->nactive; ++j) {
            const double* q = &s[(size_t)j * RES_NV];
            const int i = act[j];
            if (q[5] > 0) {
                diverged = i;
                b->active[i] = 0;
                b->iparity[i] = b->parity;
                changed = true;
                continue;
            }
            const double ru = q[1] > 0 ? std::sqrt(q[0] / q[1]) : (q[0] > 0 ? INFINITY : 0.0);
            const double rt = q[3] > 0 ? std::sqrt(q[2] / q[3]) : (q[2] > 0 ? INFINITY : 0.0);
            res[i] = (ru > rt ? ru : rt) / (double)k;
            if (res[i] <= tol) {
                b->active[i] = 0;
                b->iparity[i] = b->parity;
                changed = true;
            }
        }
        slot ^= 1;
        if (changed && (rc = batch_rebuild(b))) {
            b->active = was_active;   // the lists are as before
            return rc;
        }
        if (diverged >= 0) {
            if (steps_out) std::copy(done.begin(), done.end(), steps_out);
            if (res_out) std::copy(res.begin(), res.end(), res_out);
            return fail(LBM_ERR_DIVERGED, "instance %d holds NaN or Inf", diverged);
        }
    }
    if (steps_out) std::copy(done.begin(), done.end(), steps_out);
    if (res_out) std::copy(res.begin(), res.end(), res_out);
    return LBM_OK;
}

int lbm_batch_nusselt(lbm_batch* b, double* nu_inner, double* nu_outer) {
    if (!b || !nu_inner || !nu_outer) return fail(LBM_ERR_INVALID, "NULL argument");
    CK(cudaSetDevice(b->device));
    std::vector<int> par(b->n);
    for (int i = 0; i < b->n; ++i) par[i] = b->cur_parity(i);
    int* d_par = (int*)(b->partials);   // scratch: n ints fit in the partial rows
    CK(cudaMemcpyAsync(d_par, par.data(), b->n * sizeof(int), cudaMemcpyHostToDevice, b->stream));
    DISPATCH_STO(b->storage, k_batch_nusselt<S_><<<b->n, 256, 0, b->stream>>>(b->d_desc, b->pool, d_par, b->result));
    CK(cudaGetLastError());
    std::vector<double> r(2 * (size_t)b->n);
    CK(cudaMemcpyAsync(r.data(), b->result, r.size() * sizeof(double), cudaMemcpyDeviceToHost, b->stream));
    CK(cudaStreamSynchronize(b->stream));
    for (int i = 0; i < b->n; ++i) {
        const bool no_eq42 = b->p[i].geometry == LBM_PIPE_INFLOW || b->p[i].heater_len > 0;
        nu_inner[i] = b->p[i].geometry == LBM_PIPE_PERIODIC_Z || no_eq42 ? NAN : r[2 * i];
        nu_outer[i] = no_eq42 ? NAN : r[2 * i + 1];
    }
    return LBM_OK;
}

int lbm_batch_pipe_nusselt(lbm_batch* b, int32_t i, double* nu, int32_t nz) {
    if (!b || !nu || i < 0 || i >= b->n) return fail(LBM_ERR_INVALID, "bad batch, instance or pointer");
    if (b->p[i].geometry != LBM_PIPE_INFLOW) return fail(LBM_ERR_INVALID, "instance %d is not LBM_PIPE_INFLOW", i);
    if (nz != b->p[i].nz) return fail(LBM_ERR_INVALID, "nz = %d, instance %d has %d", nz, i, b->p[i].nz);
    CK(cudaSetDevice(b->device));
    const InstDesc& d = b->desc[i];
    float* m = b->macpool + d.off_mac;   // snapshot slot 0 of this instance as staging
    const dim3 g((unsigned)((nz + 127) / 128), (unsigned)b->p[i].nr);
    DISPATCH_STO(b->storage, k_moments<S_><<<g, 128, 0, b->stream>>>(d.c, batch_buf<S_>(b, i, b->cur_parity(i)),
                                                                      (const PP<S_>*)(b->pool + d.off_phi), d.plane,
                                                                      nullptr, nullptr, m + 2 * d.plane,
                                                                      m + 3 * d.plane));
    CK(cudaGetLastError());
    double* dn = nullptr;
    CK(cudaMallocAsync((void**)&dn, (size_t)nz * sizeof(double), b->stream));
    k_pipe_nusselt<<<(unsigned)((nz + 127) / 128), 128, 0, b->stream>>>(b->p[i].nr, nz, d.r0, m + 2 * d.plane,
                                                                        m + 3 * d.plane, dn);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(nu, dn, (size_t)nz * sizeof(double), cudaMemcpyDeviceToHost, b->stream);
    cudaFreeAsync(dn, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return fail(LBM_ERR_CUDA, "batch pipe Nusselt: %s", cudaGetErrorString(e));
    return LBM_OK;
}

int lbm_batch_moments(lbm_batch* b, int32_t i, float* rho, float* ur, float* uz, float* T, int on_device) {
    if (!b || i < 0 || i >= b->n) return fail(LBM_ERR_INVALID, "bad batch or instance");
    CK(cudaSetDevice(b->device));
    const InstDesc& d = b->desc[i];
    const int64_t N = (int64_t)b->p[i].nr * b->p[i].nz;
    float* m = b->macpool + d.off_mac;   // snapshot slot 0 of this instance as staging
    const dim3 g((unsigned)((b->p[i].nz + 127) / 128), (unsigned)b->p[i].nr);
    float* outs[4] = {rho, ur, uz, T};
    float* dst[4];
    for (int j = 0; j < 4; ++j) dst[j] = on_device ? outs[j] : (outs[j] ? m + j * d.plane : nullptr);
    const int cur = b->cur_parity(i);
    if (b->storage != LBM_F32) {
        CK(launch_fields16(b->storage, b->inst16[i], cur, dst[0], dst[1], dst[2], dst[3], b->stream));
    } else if (b->step32) {
        CK(launch_fields32(b->inst32[i].c, b->inst32[i].s[cur], b->inst32[i].phi, b->inst32[i].plane, dst[0], dst[1], dst[2],
                           dst[3], b->stream));
    } else {
        k_moments<LBM_F32><<<g, 128, 0, b->stream>>>(d.c, batch_buf<LBM_F32>(b, i, cur), (const float*)(b->pool + d.off_phi),
                                                     d.plane, dst[0], dst[1], dst[2], dst[3]);
        CK(cudaGetLastError());
    }
    if (!on_device)
        for (int j = 0; j < 4; ++j)
            if (outs[j]) CK(cudaMemcpyAsync(outs[j], dst[j], N * sizeof(float), cudaMemcpyDeviceToHost, b->stream));
    CK(cudaStreamSynchronize(b->stream));
    return LBM_OK;
}

// Autotuner: time `steps` batched steps for each bulk tile shape (columns x rows per
// block x rows per thread, at most 256 threads) and keep the fastest.  Leaves the state
// advanced by the steps it ran (2 warm-up + `steps` per shape).  Steps that launch no such
// tile (k_batch_step, k_batch_step16, staged tiles alone) time the present shape only.
static const int kTuneShapes[][3] = {{64, 1, 1}, {128, 1, 1}, {256, 1, 1}, {64, 2, 1}, {128, 2, 1}, {64, 4, 1},
                                     {32, 8, 1}, {64, 1, 2}, {64, 1, 4}, {128, 1, 2}, {128, 1, 4}, {32, 4, 4}};

int lbm_batch_set_staging(lbm_batch* b, int enable) {
    if (!b) return fail(LBM_ERR_INVALID, "batch is NULL");
    CK(cudaSetDevice(b->device));
    b->stage = enable != 0;
    return batch_rebuild(b);   // the tile lists (and the captured graph) follow the choice
}

int lbm_batch_set_wait_limit(lbm_batch* b, int rounds) {
    if (!b) return fail(LBM_ERR_INVALID, "batch is NULL");
    CK(cudaSetDevice(b->device));
    b->spin = rounds < 0 ? STAGE_SPIN : rounds;
    b->limit_set = rounds >= 0;
    return batch_rebuild(b);   // the launches (and the captured graph) follow the limit
}

int lbm_batch_wait_status(lbm_batch* b, int clear) {
    if (!b) return fail(LBM_ERR_INVALID, "batch is NULL");
    if (!b->wait_status) return LBM_OK;
    CK(cudaSetDevice(b->device));
    int v = 0;
    CK(cudaMemcpyAsync(&v, b->wait_status, sizeof(int), cudaMemcpyDeviceToHost, b->stream));
    CK(cudaStreamSynchronize(b->stream));
    if (clear && v) CK(cudaMemsetAsync(b->wait_status, 0, sizeof(int), b->stream));
    if (v == LBM_ERR_TIMEOUT)
        return fail(LBM_ERR_TIMEOUT, "a bounded wait of the staged batch kernel ran out (step results are invalid)");
    if (v) return fail(v, "the staged batch kernel was launched for an odd nz (step results are invalid)");
    return LBM_OK;
}

int lbm_batch_tune(lbm_batch* b, int32_t steps, int32_t* bz_out, int32_t* rows_out, float* ms_out) {
    if (!b || steps < 1) return fail(LBM_ERR_INVALID, "bad batch or steps");
    CK(cudaSetDevice(b->device));
    cudaEvent_t e0, e1;
    CK(cudaEventCreate(&e0));
    CK(cudaEventCreate(&e1));
    float best = INFINITY;
    int bb = b->bz, br = b->rows, bt = b->rpt;
    int rc = LBM_OK;
    std::vector<std::array<int, 3>> shapes;
    if (batch_bulk_tiles(b))
        for (const auto& s : kTuneShapes) shapes.push_back({s[0], s[1], s[2]});
    else
        shapes.push_back({bb, br, bt});
    for (const auto& s : shapes) {
        if (s != std::array<int, 3>{b->bz, b->rows, b->rpt} && (rc = batch_reshape(b, s[0], s[1], s[2]))) break;
        if ((rc = lbm_batch_step(b, 2))) break;   // warm-up
        cudaEventRecord(e0, b->stream);
        if ((rc = lbm_batch_step(b, steps))) break;
        cudaEventRecord(e1, b->stream);
        cudaEventSynchronize(e1);
        float ms = 0;
        cudaEventElapsedTime(&ms, e0, e1);
        if (ms < best) { best = ms; bb = s[0]; br = s[1]; bt = s[2]; }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc) return rc;
    if ((bb != b->bz || br != b->rows || bt != b->rpt) && (rc = batch_reshape(b, bb, br, bt))) return rc;
    if (bz_out) *bz_out = bb;
    if (rows_out) *rows_out = br * bt;
    if (ms_out) *ms_out = best / (float)steps;
    return LBM_OK;
}

int lbm_batch_get_info(lbm_batch* b, int32_t i, lbm_info* out) {
    if (!b || !out || i < 0 || i >= b->n) return fail(LBM_ERR_INVALID, "bad batch, instance or pointer");
    *out = b->info[i];
    out->steps = b->steps;
    return LBM_OK;
}

}  // extern "C"
