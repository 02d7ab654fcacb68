// GENERATED by csrc/gen_fast.py from fast/signatures.json -- do not edit.
// signature: 128|0e|3|0:0:0,0:1:1,0:2:2,0:3:3
// 128x0e (x) harmonics l<=3: P=4 D=16 nnz=16 pairs=16
#include "fast_fwd.cuh"
#include "fast_bwd.cuh"
#include "fast_launch.cuh"

namespace e3j {
namespace fast {
namespace {
__device__ const PairRec kPair_s128_l3[20] = {
    {0,1}, {1,1}, {2,1}, {3,0}, {3,1}, {4,1}, {5,1}, {6,1}, {7,1}, {8,1}, {9,1}, {10,1}, {11,1}, {12,1}, {13,1}, {14,1}, {15,1}, {16,0}, {16,0}, {16,0}};
__device__ const float kVal_s128_l3[16] = {
    1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f};
__device__ const unsigned char kI2_s128_l3[16] = {
    0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15};
__device__ const PairRec kBPair_s128_l3[24] = {
    {0,1}, {1,0}, {1,0}, {1,0}, {1,1}, {2,1}, {3,1}, {4,0}, {4,1}, {5,1}, {6,1}, {7,1}, {8,1}, {9,0}, {9,0}, {9,0}, {9,1}, {10,1}, {11,1}, {12,1}, {13,1}, {14,1}, {15,1}, {16,0}};
__device__ const float kBVal_s128_l3[16] = {
    1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f};
__device__ const unsigned char kBI2_s128_l3[16] = {
    0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15};
__device__ const unsigned char kBRow_s128_l3[28] = {
    0, 0, 0, 0, 0, 0, 0, 1, 2, 3, 3, 3, 3, 3, 4, 5, 6, 7, 8, 8, 8, 9, 10, 11, 12, 13, 14, 15};

struct Sig_s128_l3 {
    static constexpr int NQ = 128, DIN = 1, DSH = 16, P = 4, D = 16;
    static constexpr int NNZ = 16, NPAIR = 16, V = 4;
    static constexpr int FW = 4, FT = 12, FS = 2, FC = 3, F_RMAX = 5, F_APAD = 20, F_NREC = 1, F_NPMAX = 8, F_MAXREG = 255;
    // fused double backward (cotangent of grad_out): tile, stages, CTAs per SM (DFT = 0: not generated)
    static constexpr int DFT = 10, DFS = 2, DFC = 2, DFV = 4;
    using DFVec = float4;
    using Vec = float4;
    __device__ static __forceinline__ PairRec pair_rec(int i) { return kPair_s128_l3[i]; }
    __device__ static __forceinline__ float rec_val(int i) { return kVal_s128_l3[i]; }
    __device__ static __forceinline__ unsigned char rec_i2(int i) { return kI2_s128_l3[i]; }
    static constexpr int f_row0(int g) {
        switch (g) {
            case 0: return 0;
            case 1: return 3;
            case 2: return 7;
            case 3: return 11;
            case 4: return 16;
            default: return 16;
        }
    }
    static constexpr int f_a0(int g) {
        switch (g) {
            case 0: return 0;
            case 1: return 4;
            case 2: return 8;
            case 3: return 12;
            case 4: return 20;
            default: return 20;
        }
    }
    template <int G>
    __device__ static __forceinline__ void fwd_edge(Vec (&acc)[F_RMAX], const Vec* __restrict__ xs, const Vec* __restrict__ ss, const float* __restrict__ As) {
        constexpr int NQV = NQ / V;
        if constexpr (G == 0) {
            const Vec x0 = xs[0 * NQV];
            const Vec s0 = ss[0 * NQV];  // path 0: l1=0 l2=0 -> L=0
            const Vec sx0_0 = pmul(s0, x0);
            const float4 a0 = *reinterpret_cast<const float4*>(As + 0);
            pfma(acc[0], a0.x, sx0_0);
            const Vec s1 = ss[1 * NQV];  // path 1: l1=0 l2=1 -> L=1
            const Vec sx1_0 = pmul(s1, x0);
            pfma(acc[1], a0.y, sx1_0);
            pfma(acc[2], a0.z, sx1_0);
        }
        if constexpr (G == 1) {
            const Vec x0 = xs[0 * NQV];
            const Vec s1 = ss[1 * NQV];  // path 1: l1=0 l2=1 -> L=1
            const Vec sx1_0 = pmul(s1, x0);
            const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
            pfma(acc[0], a1.x, sx1_0);
            const Vec s2 = ss[2 * NQV];  // path 2: l1=0 l2=2 -> L=2
            const Vec sx2_0 = pmul(s2, x0);
            pfma(acc[1], a1.y, sx2_0);
            pfma(acc[2], a1.z, sx2_0);
            pfma(acc[3], a1.w, sx2_0);
        }
        if constexpr (G == 2) {
            const Vec x0 = xs[0 * NQV];
            const Vec s2 = ss[2 * NQV];  // path 2: l1=0 l2=2 -> L=2
            const Vec sx2_0 = pmul(s2, x0);
            const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
            pfma(acc[0], a2.x, sx2_0);
            pfma(acc[1], a2.y, sx2_0);
            const Vec s3 = ss[3 * NQV];  // path 3: l1=0 l2=3 -> L=3
            const Vec sx3_0 = pmul(s3, x0);
            pfma(acc[2], a2.z, sx3_0);
            pfma(acc[3], a2.w, sx3_0);
        }
        if constexpr (G == 3) {
            const Vec x0 = xs[0 * NQV];
            const Vec s3 = ss[3 * NQV];  // path 3: l1=0 l2=3 -> L=3
            const Vec sx3_0 = pmul(s3, x0);
            const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
            pfma(acc[0], a3.x, sx3_0);
            pfma(acc[1], a3.y, sx3_0);
            pfma(acc[2], a3.z, sx3_0);
            pfma(acc[3], a3.w, sx3_0);
            const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
            pfma(acc[4], a4.x, sx3_0);
        }
    }
    template <int G>
    __device__ static __forceinline__ void fwd2_edge(DFVec (&acc)[F_RMAX], const DFVec* __restrict__ xs, const DFVec* __restrict__ uxs, const DFVec* __restrict__ ss, const DFVec* __restrict__ uss, const float* __restrict__ As, const float* __restrict__ Bs) {
        constexpr int NQV = NQ / DFV;
        if constexpr (G == 0) {
            const DFVec x0 = xs[0 * NQV];
            const DFVec ux0 = uxs[0 * NQV];
            const DFVec s0 = ss[0 * NQV];
            const DFVec us0 = uss[0 * NQV];
            const DFVec sx0_0 = pmul(s0, x0);
            DFVec sxu0_0 = pmul(s0, ux0); pfma(sxu0_0, us0, x0);
            const float4 a0 = *reinterpret_cast<const float4*>(As + 0);
            const float4 b0 = *reinterpret_cast<const float4*>(Bs + 0);
            pfma(acc[0], a0.x, sxu0_0);
            pfma(acc[0], b0.x, sx0_0);
            const DFVec s1 = ss[1 * NQV];
            const DFVec us1 = uss[1 * NQV];
            const DFVec sx1_0 = pmul(s1, x0);
            DFVec sxu1_0 = pmul(s1, ux0); pfma(sxu1_0, us1, x0);
            pfma(acc[1], a0.y, sxu1_0);
            pfma(acc[1], b0.y, sx1_0);
            pfma(acc[2], a0.z, sxu1_0);
            pfma(acc[2], b0.z, sx1_0);
        }
        if constexpr (G == 1) {
            const DFVec x0 = xs[0 * NQV];
            const DFVec ux0 = uxs[0 * NQV];
            const DFVec s1 = ss[1 * NQV];
            const DFVec us1 = uss[1 * NQV];
            const DFVec sx1_0 = pmul(s1, x0);
            DFVec sxu1_0 = pmul(s1, ux0); pfma(sxu1_0, us1, x0);
            const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
            const float4 b1 = *reinterpret_cast<const float4*>(Bs + 4);
            pfma(acc[0], a1.x, sxu1_0);
            pfma(acc[0], b1.x, sx1_0);
            const DFVec s2 = ss[2 * NQV];
            const DFVec us2 = uss[2 * NQV];
            const DFVec sx2_0 = pmul(s2, x0);
            DFVec sxu2_0 = pmul(s2, ux0); pfma(sxu2_0, us2, x0);
            pfma(acc[1], a1.y, sxu2_0);
            pfma(acc[1], b1.y, sx2_0);
            pfma(acc[2], a1.z, sxu2_0);
            pfma(acc[2], b1.z, sx2_0);
            pfma(acc[3], a1.w, sxu2_0);
            pfma(acc[3], b1.w, sx2_0);
        }
        if constexpr (G == 2) {
            const DFVec x0 = xs[0 * NQV];
            const DFVec ux0 = uxs[0 * NQV];
            const DFVec s2 = ss[2 * NQV];
            const DFVec us2 = uss[2 * NQV];
            const DFVec sx2_0 = pmul(s2, x0);
            DFVec sxu2_0 = pmul(s2, ux0); pfma(sxu2_0, us2, x0);
            const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
            const float4 b2 = *reinterpret_cast<const float4*>(Bs + 8);
            pfma(acc[0], a2.x, sxu2_0);
            pfma(acc[0], b2.x, sx2_0);
            pfma(acc[1], a2.y, sxu2_0);
            pfma(acc[1], b2.y, sx2_0);
            const DFVec s3 = ss[3 * NQV];
            const DFVec us3 = uss[3 * NQV];
            const DFVec sx3_0 = pmul(s3, x0);
            DFVec sxu3_0 = pmul(s3, ux0); pfma(sxu3_0, us3, x0);
            pfma(acc[2], a2.z, sxu3_0);
            pfma(acc[2], b2.z, sx3_0);
            pfma(acc[3], a2.w, sxu3_0);
            pfma(acc[3], b2.w, sx3_0);
        }
        if constexpr (G == 3) {
            const DFVec x0 = xs[0 * NQV];
            const DFVec ux0 = uxs[0 * NQV];
            const DFVec s3 = ss[3 * NQV];
            const DFVec us3 = uss[3 * NQV];
            const DFVec sx3_0 = pmul(s3, x0);
            DFVec sxu3_0 = pmul(s3, ux0); pfma(sxu3_0, us3, x0);
            const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
            const float4 b3 = *reinterpret_cast<const float4*>(Bs + 12);
            pfma(acc[0], a3.x, sxu3_0);
            pfma(acc[0], b3.x, sx3_0);
            pfma(acc[1], a3.y, sxu3_0);
            pfma(acc[1], b3.y, sx3_0);
            pfma(acc[2], a3.z, sxu3_0);
            pfma(acc[2], b3.z, sx3_0);
            pfma(acc[3], a3.w, sxu3_0);
            pfma(acc[3], b3.w, sx3_0);
            const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
            const float4 b4 = *reinterpret_cast<const float4*>(Bs + 16);
            pfma(acc[4], a4.x, sxu3_0);
            pfma(acc[4], b4.x, sx3_0);
        }
    }
    // writes the group's rows to dst[r * stride] (dst already offset by the lane and the first row)
    template <int G, class VecT>
    __device__ static __forceinline__ void fwd_store(const VecT (&acc)[F_RMAX], VecT* __restrict__ dst, const int stride) {
        if constexpr (G == 0) {
            dst[0 * stride] = acc[0];
            dst[1 * stride] = acc[1];
            dst[2 * stride] = acc[2];
        }
        if constexpr (G == 1) {
            dst[0 * stride] = acc[0];
            dst[1 * stride] = acc[1];
            dst[2 * stride] = acc[2];
            dst[3 * stride] = acc[3];
        }
        if constexpr (G == 2) {
            dst[0 * stride] = acc[0];
            dst[1 * stride] = acc[1];
            dst[2 * stride] = acc[2];
            dst[3 * stride] = acc[3];
        }
        if constexpr (G == 3) {
            dst[0 * stride] = acc[0];
            dst[1 * stride] = acc[1];
            dst[2 * stride] = acc[2];
            dst[3 * stride] = acc[3];
            dst[4 * stride] = acc[4];
        }
    }
    // ---- backward: path groups [[0], [1], [2], [3]]
    static constexpr int BV = 4;  // channels per lane in the backward
    using BVec = float4;
    static constexpr int BW = 4, BT = 8, BS = 2, BC = 3, B_RMAX = 7, B_APAD = 24, B_NREC = 1;
    // edge-wise backward (one warp per edge, grad_out rows read from shared memory): edges per tile (0 = not generated), ring stages
    static constexpr int ET = 16, ES = 2, EV = 4, EXG = 0;   // EXG: sender rows not staged
    static constexpr int ST = 16;   // columns of the scheduled backward
    // the same for the standalone tensor product: rows per ring slot (0 = not generated), ring slots
    static constexpr int ETR = 0, ESR = 3;
    // fused double backward (edge outputs): edges per tile (0 = not generated), ring stages
    static constexpr int DT = 8, DS = 2, DV = 4;
    using DVec = float4;
    using EVec = float4;
    __device__ static __forceinline__ PairRec b_pair_rec(int i) { return kBPair_s128_l3[i]; }
    __device__ static __forceinline__ float b_rec_val(int i) { return kBVal_s128_l3[i]; }
    __device__ static __forceinline__ unsigned char b_rec_i2(int i) { return kBI2_s128_l3[i]; }
    // output rows of path group g: b_nrow(g) of them, the r-th is b_row(g, r)
    __device__ static __forceinline__ int b_row(int g, int r) { return kBRow_s128_l3[g * B_RMAX + r]; }
    static constexpr int b_nrow(int g) {
        switch (g) {
            case 0: return 1;
            case 1: return 3;
            case 2: return 5;
            case 3: return 7;
            default: return 0;
        }
    }
    __device__ static __forceinline__ void bwd_edge(const int G, const BVec (&dm)[B_RMAX], const BVec* __restrict__ xs, const BVec* __restrict__ ss, const float* __restrict__ As, BVec (&dxp)[DIN], float (&dyl)[16], BVec* __restrict__ gw) {
        constexpr int NQV = NQ / BV;
        switch (G) {
        case 0: {
            const BVec x0 = xs[0 * NQV];
            const BVec s0 = ss[0 * NQV];  // path 0: l1=0 l2=0 -> L=0
            const BVec sx0_0 = vmul(s0, x0);
            BVec u0_0; vzero(u0_0);
            const float4 a0 = *reinterpret_cast<const float4*>(As + 0);
            vfma(u0_0, a0.x, dm[0]);
            { const float t = vdot(sx0_0, dm[0]);
              dyl[0] = 1.0f * t;
            }
            BVec ds0 = vmul(x0, u0_0);
            if (gw) gw[0 * NQV] = ds0;
            dxp[0] = vmul(s0, u0_0);
            dyl[1] = 0.f;
            dyl[2] = 0.f;
            dyl[3] = 0.f;
            dyl[4] = 0.f;
            dyl[5] = 0.f;
            dyl[6] = 0.f;
            dyl[7] = 0.f;
            dyl[8] = 0.f;
            dyl[9] = 0.f;
            dyl[10] = 0.f;
            dyl[11] = 0.f;
            dyl[12] = 0.f;
            dyl[13] = 0.f;
            dyl[14] = 0.f;
            dyl[15] = 0.f;
        } break;
        case 1: {
            const BVec x0 = xs[0 * NQV];
            const BVec s1 = ss[1 * NQV];  // path 1: l1=0 l2=1 -> L=1
            const BVec sx1_0 = vmul(s1, x0);
            BVec u1_0; vzero(u1_0);
            const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
            vfma(u1_0, a1.x, dm[0]);
            { const float t = vdot(sx1_0, dm[0]);
              dyl[1] = 1.0f * t;
            }
            vfma(u1_0, a1.y, dm[1]);
            { const float t = vdot(sx1_0, dm[1]);
              dyl[2] = 1.0f * t;
            }
            vfma(u1_0, a1.z, dm[2]);
            { const float t = vdot(sx1_0, dm[2]);
              dyl[3] = 1.0f * t;
            }
            BVec ds1 = vmul(x0, u1_0);
            if (gw) gw[1 * NQV] = ds1;
            dxp[0] = vmul(s1, u1_0);
            dyl[0] = 0.f;
            dyl[4] = 0.f;
            dyl[5] = 0.f;
            dyl[6] = 0.f;
            dyl[7] = 0.f;
            dyl[8] = 0.f;
            dyl[9] = 0.f;
            dyl[10] = 0.f;
            dyl[11] = 0.f;
            dyl[12] = 0.f;
            dyl[13] = 0.f;
            dyl[14] = 0.f;
            dyl[15] = 0.f;
        } break;
        case 2: {
            const BVec x0 = xs[0 * NQV];
            const BVec s2 = ss[2 * NQV];  // path 2: l1=0 l2=2 -> L=2
            const BVec sx2_0 = vmul(s2, x0);
            BVec u2_0; vzero(u2_0);
            const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
            vfma(u2_0, a2.x, dm[0]);
            { const float t = vdot(sx2_0, dm[0]);
              dyl[4] = 1.0f * t;
            }
            vfma(u2_0, a2.y, dm[1]);
            { const float t = vdot(sx2_0, dm[1]);
              dyl[5] = 1.0f * t;
            }
            vfma(u2_0, a2.z, dm[2]);
            { const float t = vdot(sx2_0, dm[2]);
              dyl[6] = 1.0f * t;
            }
            vfma(u2_0, a2.w, dm[3]);
            { const float t = vdot(sx2_0, dm[3]);
              dyl[7] = 1.0f * t;
            }
            const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
            vfma(u2_0, a3.x, dm[4]);
            { const float t = vdot(sx2_0, dm[4]);
              dyl[8] = 1.0f * t;
            }
            BVec ds2 = vmul(x0, u2_0);
            if (gw) gw[2 * NQV] = ds2;
            dxp[0] = vmul(s2, u2_0);
            dyl[0] = 0.f;
            dyl[1] = 0.f;
            dyl[2] = 0.f;
            dyl[3] = 0.f;
            dyl[9] = 0.f;
            dyl[10] = 0.f;
            dyl[11] = 0.f;
            dyl[12] = 0.f;
            dyl[13] = 0.f;
            dyl[14] = 0.f;
            dyl[15] = 0.f;
        } break;
        case 3: {
            const BVec x0 = xs[0 * NQV];
            const BVec s3 = ss[3 * NQV];  // path 3: l1=0 l2=3 -> L=3
            const BVec sx3_0 = vmul(s3, x0);
            BVec u3_0; vzero(u3_0);
            const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
            vfma(u3_0, a4.x, dm[0]);
            { const float t = vdot(sx3_0, dm[0]);
              dyl[9] = 1.0f * t;
            }
            vfma(u3_0, a4.y, dm[1]);
            { const float t = vdot(sx3_0, dm[1]);
              dyl[10] = 1.0f * t;
            }
            vfma(u3_0, a4.z, dm[2]);
            { const float t = vdot(sx3_0, dm[2]);
              dyl[11] = 1.0f * t;
            }
            vfma(u3_0, a4.w, dm[3]);
            { const float t = vdot(sx3_0, dm[3]);
              dyl[12] = 1.0f * t;
            }
            const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
            vfma(u3_0, a5.x, dm[4]);
            { const float t = vdot(sx3_0, dm[4]);
              dyl[13] = 1.0f * t;
            }
            vfma(u3_0, a5.y, dm[5]);
            { const float t = vdot(sx3_0, dm[5]);
              dyl[14] = 1.0f * t;
            }
            vfma(u3_0, a5.z, dm[6]);
            { const float t = vdot(sx3_0, dm[6]);
              dyl[15] = 1.0f * t;
            }
            BVec ds3 = vmul(x0, u3_0);
            if (gw) gw[3 * NQV] = ds3;
            dxp[0] = vmul(s3, u3_0);
            dyl[0] = 0.f;
            dyl[1] = 0.f;
            dyl[2] = 0.f;
            dyl[3] = 0.f;
            dyl[4] = 0.f;
            dyl[5] = 0.f;
            dyl[6] = 0.f;
            dyl[7] = 0.f;
            dyl[8] = 0.f;
        } break;
        default: {
#pragma unroll
            for (int i = 0; i < DIN; ++i) vzero(dxp[i]);
#pragma unroll
            for (int i = 0; i < 16; ++i) dyl[i] = 0.f;
        } break;
        }
    }
    __device__ static __forceinline__ void bwd_edge_all(const EVec* __restrict__ dms, const EVec* __restrict__ xs, const EVec* __restrict__ ss, const float* __restrict__ As, EVec (&dxp)[DIN], float (&dyl)[16], EVec* __restrict__ gw) {
        constexpr int NQV = NQ / EV;
        const EVec x0 = xs[0 * NQV];
        const EVec s0 = ss[0 * NQV];  // path 0: l1=0 l2=0 -> L=0
        const EVec sx0_0 = vmul(s0, x0);
        EVec u0_0; vzero(u0_0);
        const EVec d0_0 = dms[0 * NQV];
        const float4 a0 = *reinterpret_cast<const float4*>(As + 0);
        vfma(u0_0, a0.x, d0_0);
        { const float t = vdot(sx0_0, d0_0);
          dyl[0] = 1.0f * t;
        }
        EVec ds0 = vmul(x0, u0_0);
        if (gw) gw[0 * NQV] = ds0;
        dxp[0] = vmul(s0, u0_0);
        const EVec s1 = ss[1 * NQV];  // path 1: l1=0 l2=1 -> L=1
        const EVec sx1_0 = vmul(s1, x0);
        EVec u1_0; vzero(u1_0);
        const EVec d1_1 = dms[1 * NQV];
        const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
        vfma(u1_0, a1.x, d1_1);
        { const float t = vdot(sx1_0, d1_1);
          dyl[1] = 1.0f * t;
        }
        const EVec d1_2 = dms[2 * NQV];
        vfma(u1_0, a1.y, d1_2);
        { const float t = vdot(sx1_0, d1_2);
          dyl[2] = 1.0f * t;
        }
        const EVec d1_3 = dms[3 * NQV];
        vfma(u1_0, a1.z, d1_3);
        { const float t = vdot(sx1_0, d1_3);
          dyl[3] = 1.0f * t;
        }
        EVec ds1 = vmul(x0, u1_0);
        if (gw) gw[1 * NQV] = ds1;
        vfma(dxp[0], s1, u1_0);
        const EVec s2 = ss[2 * NQV];  // path 2: l1=0 l2=2 -> L=2
        const EVec sx2_0 = vmul(s2, x0);
        EVec u2_0; vzero(u2_0);
        const EVec d2_4 = dms[4 * NQV];
        const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
        vfma(u2_0, a2.x, d2_4);
        { const float t = vdot(sx2_0, d2_4);
          dyl[4] = 1.0f * t;
        }
        const EVec d2_5 = dms[5 * NQV];
        vfma(u2_0, a2.y, d2_5);
        { const float t = vdot(sx2_0, d2_5);
          dyl[5] = 1.0f * t;
        }
        const EVec d2_6 = dms[6 * NQV];
        vfma(u2_0, a2.z, d2_6);
        { const float t = vdot(sx2_0, d2_6);
          dyl[6] = 1.0f * t;
        }
        const EVec d2_7 = dms[7 * NQV];
        vfma(u2_0, a2.w, d2_7);
        { const float t = vdot(sx2_0, d2_7);
          dyl[7] = 1.0f * t;
        }
        const EVec d2_8 = dms[8 * NQV];
        const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
        vfma(u2_0, a3.x, d2_8);
        { const float t = vdot(sx2_0, d2_8);
          dyl[8] = 1.0f * t;
        }
        EVec ds2 = vmul(x0, u2_0);
        if (gw) gw[2 * NQV] = ds2;
        vfma(dxp[0], s2, u2_0);
        const EVec s3 = ss[3 * NQV];  // path 3: l1=0 l2=3 -> L=3
        const EVec sx3_0 = vmul(s3, x0);
        EVec u3_0; vzero(u3_0);
        const EVec d3_9 = dms[9 * NQV];
        const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
        vfma(u3_0, a4.x, d3_9);
        { const float t = vdot(sx3_0, d3_9);
          dyl[9] = 1.0f * t;
        }
        const EVec d3_10 = dms[10 * NQV];
        vfma(u3_0, a4.y, d3_10);
        { const float t = vdot(sx3_0, d3_10);
          dyl[10] = 1.0f * t;
        }
        const EVec d3_11 = dms[11 * NQV];
        vfma(u3_0, a4.z, d3_11);
        { const float t = vdot(sx3_0, d3_11);
          dyl[11] = 1.0f * t;
        }
        const EVec d3_12 = dms[12 * NQV];
        vfma(u3_0, a4.w, d3_12);
        { const float t = vdot(sx3_0, d3_12);
          dyl[12] = 1.0f * t;
        }
        const EVec d3_13 = dms[13 * NQV];
        const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
        vfma(u3_0, a5.x, d3_13);
        { const float t = vdot(sx3_0, d3_13);
          dyl[13] = 1.0f * t;
        }
        const EVec d3_14 = dms[14 * NQV];
        vfma(u3_0, a5.y, d3_14);
        { const float t = vdot(sx3_0, d3_14);
          dyl[14] = 1.0f * t;
        }
        const EVec d3_15 = dms[15 * NQV];
        vfma(u3_0, a5.z, d3_15);
        { const float t = vdot(sx3_0, d3_15);
          dyl[15] = 1.0f * t;
        }
        EVec ds3 = vmul(x0, u3_0);
        if (gw) gw[3 * NQV] = ds3;
        vfma(dxp[0], s3, u3_0);
    }
    __device__ static __forceinline__ void bwd2_edge_all(const DVec* __restrict__ dms, const DVec* __restrict__ xs, const DVec* __restrict__ uxs, const DVec* __restrict__ ss, const DVec* __restrict__ uss, const float* __restrict__ As, const float* __restrict__ Bs, DVec (&dxp)[DIN], float (&dyl)[16], DVec* __restrict__ gw) {
        constexpr int NQV = NQ / DV;
        const DVec x0 = xs[0 * NQV];
        const DVec ux0 = uxs[0 * NQV];
        const DVec s0 = ss[0 * NQV];  // path 0: l1=0 l2=0 -> L=0
        const DVec us0 = uss[0 * NQV];
        DVec sxu0_0 = pmul(s0, ux0); pfma(sxu0_0, us0, x0);
        DVec v0_0; vzero(v0_0);
        DVec w0_0; vzero(w0_0);
        const DVec d0_0 = dms[0 * NQV];
        const float4 a0 = *reinterpret_cast<const float4*>(As + 0);
        const float4 b0 = *reinterpret_cast<const float4*>(Bs + 0);
        pfma(v0_0, a0.x, d0_0);
        pfma(w0_0, b0.x, d0_0);
        { const float t = vdot(sxu0_0, d0_0);
          dyl[0] = 1.0f * t;
        }
        DVec ds0 = pmul(ux0, v0_0); pfma(ds0, x0, w0_0);
        if (gw) gw[0 * NQV] = ds0;
        dxp[0] = pmul(us0, v0_0); pfma(dxp[0], s0, w0_0);
        const DVec s1 = ss[1 * NQV];  // path 1: l1=0 l2=1 -> L=1
        const DVec us1 = uss[1 * NQV];
        DVec sxu1_0 = pmul(s1, ux0); pfma(sxu1_0, us1, x0);
        DVec v1_0; vzero(v1_0);
        DVec w1_0; vzero(w1_0);
        const DVec d1_1 = dms[1 * NQV];
        const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
        const float4 b1 = *reinterpret_cast<const float4*>(Bs + 4);
        pfma(v1_0, a1.x, d1_1);
        pfma(w1_0, b1.x, d1_1);
        { const float t = vdot(sxu1_0, d1_1);
          dyl[1] = 1.0f * t;
        }
        const DVec d1_2 = dms[2 * NQV];
        pfma(v1_0, a1.y, d1_2);
        pfma(w1_0, b1.y, d1_2);
        { const float t = vdot(sxu1_0, d1_2);
          dyl[2] = 1.0f * t;
        }
        const DVec d1_3 = dms[3 * NQV];
        pfma(v1_0, a1.z, d1_3);
        pfma(w1_0, b1.z, d1_3);
        { const float t = vdot(sxu1_0, d1_3);
          dyl[3] = 1.0f * t;
        }
        DVec ds1 = pmul(ux0, v1_0); pfma(ds1, x0, w1_0);
        if (gw) gw[1 * NQV] = ds1;
        pfma(dxp[0], us1, v1_0); pfma(dxp[0], s1, w1_0);
        const DVec s2 = ss[2 * NQV];  // path 2: l1=0 l2=2 -> L=2
        const DVec us2 = uss[2 * NQV];
        DVec sxu2_0 = pmul(s2, ux0); pfma(sxu2_0, us2, x0);
        DVec v2_0; vzero(v2_0);
        DVec w2_0; vzero(w2_0);
        const DVec d2_4 = dms[4 * NQV];
        const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
        const float4 b2 = *reinterpret_cast<const float4*>(Bs + 8);
        pfma(v2_0, a2.x, d2_4);
        pfma(w2_0, b2.x, d2_4);
        { const float t = vdot(sxu2_0, d2_4);
          dyl[4] = 1.0f * t;
        }
        const DVec d2_5 = dms[5 * NQV];
        pfma(v2_0, a2.y, d2_5);
        pfma(w2_0, b2.y, d2_5);
        { const float t = vdot(sxu2_0, d2_5);
          dyl[5] = 1.0f * t;
        }
        const DVec d2_6 = dms[6 * NQV];
        pfma(v2_0, a2.z, d2_6);
        pfma(w2_0, b2.z, d2_6);
        { const float t = vdot(sxu2_0, d2_6);
          dyl[6] = 1.0f * t;
        }
        const DVec d2_7 = dms[7 * NQV];
        pfma(v2_0, a2.w, d2_7);
        pfma(w2_0, b2.w, d2_7);
        { const float t = vdot(sxu2_0, d2_7);
          dyl[7] = 1.0f * t;
        }
        const DVec d2_8 = dms[8 * NQV];
        const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
        const float4 b3 = *reinterpret_cast<const float4*>(Bs + 12);
        pfma(v2_0, a3.x, d2_8);
        pfma(w2_0, b3.x, d2_8);
        { const float t = vdot(sxu2_0, d2_8);
          dyl[8] = 1.0f * t;
        }
        DVec ds2 = pmul(ux0, v2_0); pfma(ds2, x0, w2_0);
        if (gw) gw[2 * NQV] = ds2;
        pfma(dxp[0], us2, v2_0); pfma(dxp[0], s2, w2_0);
        const DVec s3 = ss[3 * NQV];  // path 3: l1=0 l2=3 -> L=3
        const DVec us3 = uss[3 * NQV];
        DVec sxu3_0 = pmul(s3, ux0); pfma(sxu3_0, us3, x0);
        DVec v3_0; vzero(v3_0);
        DVec w3_0; vzero(w3_0);
        const DVec d3_9 = dms[9 * NQV];
        const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
        const float4 b4 = *reinterpret_cast<const float4*>(Bs + 16);
        pfma(v3_0, a4.x, d3_9);
        pfma(w3_0, b4.x, d3_9);
        { const float t = vdot(sxu3_0, d3_9);
          dyl[9] = 1.0f * t;
        }
        const DVec d3_10 = dms[10 * NQV];
        pfma(v3_0, a4.y, d3_10);
        pfma(w3_0, b4.y, d3_10);
        { const float t = vdot(sxu3_0, d3_10);
          dyl[10] = 1.0f * t;
        }
        const DVec d3_11 = dms[11 * NQV];
        pfma(v3_0, a4.z, d3_11);
        pfma(w3_0, b4.z, d3_11);
        { const float t = vdot(sxu3_0, d3_11);
          dyl[11] = 1.0f * t;
        }
        const DVec d3_12 = dms[12 * NQV];
        pfma(v3_0, a4.w, d3_12);
        pfma(w3_0, b4.w, d3_12);
        { const float t = vdot(sxu3_0, d3_12);
          dyl[12] = 1.0f * t;
        }
        const DVec d3_13 = dms[13 * NQV];
        const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
        const float4 b5 = *reinterpret_cast<const float4*>(Bs + 20);
        pfma(v3_0, a5.x, d3_13);
        pfma(w3_0, b5.x, d3_13);
        { const float t = vdot(sxu3_0, d3_13);
          dyl[13] = 1.0f * t;
        }
        const DVec d3_14 = dms[14 * NQV];
        pfma(v3_0, a5.y, d3_14);
        pfma(w3_0, b5.y, d3_14);
        { const float t = vdot(sxu3_0, d3_14);
          dyl[14] = 1.0f * t;
        }
        const DVec d3_15 = dms[15 * NQV];
        pfma(v3_0, a5.z, d3_15);
        pfma(w3_0, b5.z, d3_15);
        { const float t = vdot(sxu3_0, d3_15);
          dyl[15] = 1.0f * t;
        }
        DVec ds3 = pmul(ux0, v3_0); pfma(ds3, x0, w3_0);
        if (gw) gw[3 * NQV] = ds3;
        pfma(dxp[0], us3, v3_0); pfma(dxp[0], s3, w3_0);
    }
};
}  // namespace
}  // namespace fast

extern const FastKernels kFast_s128_l3;
const FastKernels kFast_s128_l3 = {
    "128|0e|3|0:0:0,0:1:1,0:2:2,0:3:3",
    &fast::fwd_scratch_bytes<fast::Sig_s128_l3>, &fast::bwd_scratch_bytes<fast::Sig_s128_l3>, &fast::launch_fwd<fast::Sig_s128_l3>, &fast::launch_bwd<fast::Sig_s128_l3>, &fast::launch_tp_fwd<fast::Sig_s128_l3>, &fast::launch_tp_bwd<fast::Sig_s128_l3>,
    &fast::launch_dbl_edges<fast::Sig_s128_l3>, &fast::launch_dbl_out<fast::Sig_s128_l3>, nullptr, nullptr, 0};
}  // namespace e3j
