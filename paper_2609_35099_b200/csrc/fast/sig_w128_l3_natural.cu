// GENERATED by csrc/gen_fast.py from fast/signatures.json -- do not edit.
// signature: 128|0e+1o|3|0:0:0,1:1:0,0:1:1,1:0:1,1:2:1,0:2:2,1:1:2,1:3:2,0:3:3,1:2:3
// 128x0e+128x1o (x) harmonics l<=3: P=10 D=40 nnz=86 pairs=76
#include "fast_fwd.cuh"
#include "fast_bwd.cuh"
#include "fast_launch.cuh"
#include "fast_bwd1s.cuh"

namespace e3j {
namespace fast {
namespace {
__device__ const PairRec kPair_w128_l3_natural[84] = {
    {0,1}, {1,1}, {2,1}, {3,1}, {4,1}, {5,1}, {6,1}, {7,1}, {8,1}, {9,1}, {10,2}, {12,1}, {13,1}, {14,0}, {14,0}, {14,0}, {14,1}, {15,1}, {16,1}, {17,1}, {18,1}, {19,2}, {21,1}, {22,1}, {23,1}, {24,1}, {25,1}, {26,1}, {27,1}, {28,1}, {29,1}, {30,1}, {31,1}, {32,1}, {33,1}, {34,1}, {35,1}, {36,1}, {37,2}, {39,1}, {40,2}, {42,2}, {44,1}, {45,1}, {46,1}, {47,1}, {48,1}, {49,1}, {50,1}, {51,2}, {53,2}, {55,1}, {56,2}, {58,1}, {59,1}, {60,1}, {61,1}, {62,0}, {62,0}, {62,0}, {62,1}, {63,1}, {64,1}, {65,1}, {66,1}, {67,1}, {68,1}, {69,1}, {70,2}, {72,1}, {73,1}, {74,1}, {75,1}, {76,1}, {77,1}, {78,1}, {79,2}, {81,1}, {82,1}, {83,1}, {84,1}, {85,1}, {86,0}, {86,0}};
__device__ const float kVal_w128_l3_natural[86] = {
    1.0f, 0.577350259f, 0.577350259f, 0.577350259f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 0.316227764f, 0.547722578f, -0.547722578f, -0.547722578f, -0.547722578f, -0.632455528f, -0.547722578f, -0.547722578f, -0.547722578f, 0.316227764f, -0.547722578f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 0.707106769f, 0.707106769f, 0.707106769f, 0.707106769f, -0.408248305f, 0.816496611f, -0.408248305f, 0.707106769f, 0.707106769f, -0.707106769f, 0.707106769f, 0.154303357f, 0.597614288f, -0.487950027f, -0.597614288f, 0.154303357f, 0.377964467f, 0.487950027f, -0.617213428f, -0.487950027f, -0.534522474f, -0.654653668f, -0.534522474f, -0.487950027f, -0.617213428f, 0.377964467f, -0.487950027f, -0.597614288f, -0.154303357f, -0.487950027f, 0.154303357f, -0.597614288f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 0.707106769f, 0.707106769f, 0.577350259f, 0.577350259f, 0.577350259f, 0.632455528f, 0.182574183f, 0.730296731f, -0.182574183f, -0.44721359f, 0.774596691f, -0.44721359f, -0.182574183f, 0.730296731f, 0.632455528f, -0.182574183f, -0.577350259f, 0.577350259f, 0.577350259f, -0.707106769f, 0.707106769f};
__device__ const unsigned char kI2_w128_l3_natural[86] = {
    0, 1, 2, 3, 1, 2, 3, 0, 0, 0, 6, 8, 5, 4, 5, 6, 7, 4, 7, 6, 8, 4, 5, 6, 7, 8, 3, 1, 2, 1, 1, 2, 3, 3, 2, 1, 3, 13, 15, 10, 9, 11, 12, 14, 11, 10, 11, 12, 13, 10, 13, 12, 14, 9, 11, 14, 13, 15, 9, 10, 11, 12, 13, 14, 15, 8, 4, 7, 4, 5, 6, 8, 5, 4, 5, 6, 7, 4, 7, 6, 8, 5, 8, 7, 4, 8};
__device__ const PairRec kBPair_w128_l3_natural[84] = {
    {0,1}, {1,1}, {2,1}, {3,1}, {4,1}, {5,1}, {6,1}, {7,1}, {8,1}, {9,1}, {10,1}, {11,1}, {12,1}, {13,1}, {14,1}, {15,1}, {16,1}, {17,0}, {17,0}, {17,0}, {17,1}, {18,1}, {19,1}, {20,1}, {21,1}, {22,1}, {23,2}, {25,1}, {26,1}, {27,1}, {28,1}, {29,1}, {30,1}, {31,1}, {32,2}, {34,0}, {34,1}, {35,1}, {36,1}, {37,1}, {38,1}, {39,1}, {40,1}, {41,1}, {42,2}, {44,1}, {45,1}, {46,1}, {47,1}, {48,1}, {49,1}, {50,1}, {51,2}, {53,1}, {54,1}, {55,1}, {56,1}, {57,1}, {58,0}, {58,0}, {58,2}, {60,1}, {61,2}, {63,2}, {65,1}, {66,1}, {67,1}, {68,1}, {69,1}, {70,1}, {71,1}, {72,2}, {74,2}, {76,1}, {77,2}, {79,1}, {80,1}, {81,1}, {82,1}, {83,1}, {84,1}, {85,1}, {86,0}, {86,0}};
__device__ const float kBVal_w128_l3_natural[86] = {
    1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 0.707106769f, 0.707106769f, 0.707106769f, 0.707106769f, -0.408248305f, 0.816496611f, -0.408248305f, 0.707106769f, 0.707106769f, -0.707106769f, 0.707106769f, 0.577350259f, 0.577350259f, 0.577350259f, 1.0f, 1.0f, 1.0f, 0.316227764f, 0.547722578f, -0.547722578f, -0.547722578f, -0.547722578f, -0.632455528f, -0.547722578f, -0.547722578f, -0.547722578f, 0.316227764f, -0.547722578f, 1.0f, 1.0f, 1.0f, 0.707106769f, 0.707106769f, 0.577350259f, 0.577350259f, 0.577350259f, 0.632455528f, 0.182574183f, 0.730296731f, -0.182574183f, -0.44721359f, 0.774596691f, -0.44721359f, -0.182574183f, 0.730296731f, 0.632455528f, -0.182574183f, -0.577350259f, 0.577350259f, 0.577350259f, -0.707106769f, 0.707106769f, 0.154303357f, 0.597614288f, -0.487950027f, -0.597614288f, 0.154303357f, 0.377964467f, 0.487950027f, -0.617213428f, -0.487950027f, -0.534522474f, -0.654653668f, -0.534522474f, -0.487950027f, -0.617213428f, 0.377964467f, -0.487950027f, -0.597614288f, -0.154303357f, -0.487950027f, 0.154303357f, -0.597614288f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f};
__device__ const unsigned char kBI2_w128_l3_natural[86] = {
    0, 4, 5, 6, 7, 8, 3, 1, 2, 1, 1, 2, 3, 3, 2, 1, 3, 1, 2, 3, 0, 0, 0, 6, 8, 5, 4, 5, 6, 7, 4, 7, 6, 8, 1, 2, 3, 8, 4, 7, 4, 5, 6, 8, 5, 4, 5, 6, 7, 4, 7, 6, 8, 5, 8, 7, 4, 8, 13, 15, 10, 9, 11, 12, 14, 11, 10, 11, 12, 13, 10, 13, 12, 14, 9, 11, 14, 13, 15, 9, 10, 11, 12, 13, 14, 15};
__device__ const unsigned char kBRow_w128_l3_natural[48] = {
    0, 11, 12, 13, 14, 15, 16, 17, 18, 19, 20, 20, 1, 5, 6, 7, 8, 9, 10, 10, 10, 10, 10, 10, 2, 3, 4, 33, 34, 35, 36, 37, 38, 39, 39, 39, 21, 22, 23, 24, 25, 26, 27, 28, 29, 30, 31, 32};

struct Sig_w128_l3_natural {
    static constexpr int NQ = 128, DIN = 4, DSH = 16, P = 10, D = 40;
    static constexpr int NNZ = 86, NPAIR = 76, V = 4;
    static constexpr int FW = 4, FT = 7, FS = 2, FC = 2, F_RMAX = 11, F_APAD = 84, F_NREC = 2, F_NPMAX = 24, F_MAXREG = 255;
    // fused double backward (cotangent of grad_out): tile, stages, CTAs per SM (DFT = 0: not generated)
    static constexpr int DFT = 3, DFS = 2, DFC = 2, DFV = 2;
    using DFVec = float2;
    using Vec = float4;
    __device__ static __forceinline__ PairRec pair_rec(int i) { return kPair_w128_l3_natural[i]; }
    __device__ static __forceinline__ float rec_val(int i) { return kVal_w128_l3_natural[i]; }
    __device__ static __forceinline__ unsigned char rec_i2(int i) { return kI2_w128_l3_natural[i]; }
    static constexpr int f_row0(int g) {
        switch (g) {
            case 0: return 0;
            case 1: return 9;
            case 2: return 20;
            case 3: return 30;
            case 4: return 40;
            default: return 40;
        }
    }
    static constexpr int f_a0(int g) {
        switch (g) {
            case 0: return 0;
            case 1: return 16;
            case 2: return 36;
            case 3: return 60;
            case 4: return 84;
            default: return 84;
        }
    }
    template <int G>
    __device__ static __forceinline__ void fwd_edge(Vec (&acc)[F_RMAX], const Vec* __restrict__ xs, const Vec* __restrict__ ss, const float* __restrict__ As) {
        constexpr int NQV = NQ / V;
        if constexpr (G == 0) {
            const Vec x0 = xs[0 * NQV];
            const Vec x1 = xs[1 * NQV];
            const Vec x2 = xs[2 * NQV];
            const Vec x3 = xs[3 * NQV];
            const Vec s0 = ss[0 * NQV];  // path 0: l1=0 l2=0 -> L=0
            const Vec sx0_0 = pmul(s0, x0);
            const float4 a0 = *reinterpret_cast<const float4*>(As + 0);
            pfma(acc[0], a0.x, sx0_0);
            const Vec s1 = ss[1 * NQV];  // path 1: l1=1 l2=1 -> L=0
            const Vec sx1_1 = pmul(s1, x1);
            const Vec sx1_2 = pmul(s1, x2);
            const Vec sx1_3 = pmul(s1, x3);
            pfma(acc[1], a0.y, sx1_1);
            pfma(acc[1], a0.z, sx1_2);
            pfma(acc[1], a0.w, sx1_3);
            const Vec s2 = ss[2 * NQV];  // path 2: l1=0 l2=1 -> L=1
            const Vec sx2_0 = pmul(s2, x0);
            const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
            pfma(acc[2], a1.x, sx2_0);
            pfma(acc[3], a1.y, sx2_0);
            pfma(acc[4], a1.z, sx2_0);
            const Vec s3 = ss[3 * NQV];  // path 3: l1=1 l2=0 -> L=1
            const Vec sx3_1 = pmul(s3, x1);
            const Vec sx3_2 = pmul(s3, x2);
            const Vec sx3_3 = pmul(s3, x3);
            pfma(acc[5], a1.w, sx3_1);
            const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
            pfma(acc[6], a2.x, sx3_2);
            pfma(acc[7], a2.y, sx3_3);
            const Vec s4 = ss[4 * NQV];  // path 4: l1=1 l2=2 -> L=1
            const Vec sx4_1 = pmul(s4, x1);
            const Vec sx4_2 = pmul(s4, x2);
            const Vec sx4_3 = pmul(s4, x3);
            pfma(acc[8], a2.z, sx4_1);
            pfma(acc[8], a2.w, sx4_2);
            const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
            pfma(acc[8], a3.x, sx4_3);
        }
        if constexpr (G == 1) {
            const Vec x0 = xs[0 * NQV];
            const Vec x1 = xs[1 * NQV];
            const Vec x2 = xs[2 * NQV];
            const Vec x3 = xs[3 * NQV];
            const Vec s4 = ss[4 * NQV];  // path 4: l1=1 l2=2 -> L=1
            const Vec sx4_1 = pmul(s4, x1);
            const Vec sx4_2 = pmul(s4, x2);
            const Vec sx4_3 = pmul(s4, x3);
            const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
            pfma(acc[0], a4.x, sx4_1);
            pfma(acc[1], a4.w, sx4_1);
            pfma(acc[0], a4.y, sx4_2);
            const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
            pfma(acc[1], a5.x, sx4_2);
            pfma(acc[0], a4.z, sx4_3);
            pfma(acc[1], a5.y, sx4_3);
            const Vec s5 = ss[5 * NQV];  // path 5: l1=0 l2=2 -> L=2
            const Vec sx5_0 = pmul(s5, x0);
            pfma(acc[2], a5.z, sx5_0);
            pfma(acc[3], a5.w, sx5_0);
            const float4 a6 = *reinterpret_cast<const float4*>(As + 24);
            pfma(acc[4], a6.x, sx5_0);
            pfma(acc[5], a6.y, sx5_0);
            pfma(acc[6], a6.z, sx5_0);
            const Vec s6 = ss[6 * NQV];  // path 6: l1=1 l2=1 -> L=2
            const Vec sx6_1 = pmul(s6, x1);
            const Vec sx6_2 = pmul(s6, x2);
            const Vec sx6_3 = pmul(s6, x3);
            pfma(acc[7], a6.w, sx6_1);
            const float4 a7 = *reinterpret_cast<const float4*>(As + 28);
            pfma(acc[8], a7.y, sx6_1);
            pfma(acc[9], a7.w, sx6_1);
            const float4 a8 = *reinterpret_cast<const float4*>(As + 32);
            pfma(acc[10], a8.z, sx6_2);
            pfma(acc[7], a7.x, sx6_3);
            pfma(acc[8], a7.z, sx6_2);
            pfma(acc[9], a8.x, sx6_2);
            pfma(acc[10], a8.w, sx6_3);
            pfma(acc[9], a8.y, sx6_3);
        }
        if constexpr (G == 2) {
            const Vec x0 = xs[0 * NQV];
            const Vec x1 = xs[1 * NQV];
            const Vec x2 = xs[2 * NQV];
            const Vec x3 = xs[3 * NQV];
            const Vec s6 = ss[6 * NQV];  // path 6: l1=1 l2=1 -> L=2
            const Vec sx6_1 = pmul(s6, x1);
            const Vec sx6_3 = pmul(s6, x3);
            const float4 a9 = *reinterpret_cast<const float4*>(As + 36);
            pfma(acc[0], a9.x, sx6_1);
            pfma(acc[0], a9.y, sx6_3);
            const Vec s7 = ss[7 * NQV];  // path 7: l1=1 l2=3 -> L=2
            const Vec sx7_1 = pmul(s7, x1);
            const Vec sx7_2 = pmul(s7, x2);
            const Vec sx7_3 = pmul(s7, x3);
            pfma(acc[1], a9.z, sx7_1);
            const float4 a10 = *reinterpret_cast<const float4*>(As + 40);
            pfma(acc[2], a10.y, sx7_1);
            const float4 a11 = *reinterpret_cast<const float4*>(As + 44);
            pfma(acc[3], a11.x, sx7_1);
            pfma(acc[4], a11.w, sx7_1);
            const float4 a12 = *reinterpret_cast<const float4*>(As + 48);
            pfma(acc[5], a12.z, sx7_1);
            pfma(acc[1], a9.w, sx7_2);
            pfma(acc[2], a10.z, sx7_2);
            pfma(acc[3], a11.y, sx7_2);
            pfma(acc[4], a12.x, sx7_2);
            pfma(acc[5], a12.w, sx7_2);
            pfma(acc[1], a10.x, sx7_3);
            pfma(acc[2], a10.w, sx7_3);
            pfma(acc[3], a11.z, sx7_3);
            pfma(acc[4], a12.y, sx7_3);
            const float4 a13 = *reinterpret_cast<const float4*>(As + 52);
            pfma(acc[5], a13.x, sx7_3);
            const Vec s8 = ss[8 * NQV];  // path 8: l1=0 l2=3 -> L=3
            const Vec sx8_0 = pmul(s8, x0);
            pfma(acc[6], a13.y, sx8_0);
            pfma(acc[7], a13.z, sx8_0);
            pfma(acc[8], a13.w, sx8_0);
            const float4 a14 = *reinterpret_cast<const float4*>(As + 56);
            pfma(acc[9], a14.x, sx8_0);
        }
        if constexpr (G == 3) {
            const Vec x0 = xs[0 * NQV];
            const Vec x1 = xs[1 * NQV];
            const Vec x2 = xs[2 * NQV];
            const Vec x3 = xs[3 * NQV];
            const Vec s8 = ss[8 * NQV];  // path 8: l1=0 l2=3 -> L=3
            const Vec sx8_0 = pmul(s8, x0);
            const float4 a15 = *reinterpret_cast<const float4*>(As + 60);
            pfma(acc[0], a15.x, sx8_0);
            pfma(acc[1], a15.y, sx8_0);
            pfma(acc[2], a15.z, sx8_0);
            const Vec s9 = ss[9 * NQV];  // path 9: l1=1 l2=2 -> L=3
            const Vec sx9_1 = pmul(s9, x1);
            const Vec sx9_2 = pmul(s9, x2);
            const Vec sx9_3 = pmul(s9, x3);
            pfma(acc[3], a15.w, sx9_1);
            const float4 a16 = *reinterpret_cast<const float4*>(As + 64);
            pfma(acc[4], a16.y, sx9_1);
            const float4 a17 = *reinterpret_cast<const float4*>(As + 68);
            pfma(acc[5], a17.x, sx9_1);
            pfma(acc[6], a17.w, sx9_1);
            const float4 a18 = *reinterpret_cast<const float4*>(As + 72);
            pfma(acc[7], a18.z, sx9_1);
            const float4 a19 = *reinterpret_cast<const float4*>(As + 76);
            pfma(acc[8], a19.y, sx9_1);
            const float4 a20 = *reinterpret_cast<const float4*>(As + 80);
            pfma(acc[9], a20.x, sx9_1);
            pfma(acc[3], a16.x, sx9_3);
            pfma(acc[4], a16.z, sx9_2);
            pfma(acc[5], a17.y, sx9_2);
            pfma(acc[6], a18.x, sx9_2);
            pfma(acc[7], a18.w, sx9_2);
            pfma(acc[8], a19.z, sx9_2);
            pfma(acc[9], a20.y, sx9_3);
            pfma(acc[4], a16.w, sx9_3);
            pfma(acc[5], a17.z, sx9_3);
            pfma(acc[6], a18.y, sx9_3);
            pfma(acc[7], a19.x, sx9_3);
            pfma(acc[8], a19.w, sx9_3);
        }
    }
    template <int G>
    __device__ static __forceinline__ void fwd2_edge(DFVec (&acc)[F_RMAX], const DFVec* __restrict__ xs, const DFVec* __restrict__ uxs, const DFVec* __restrict__ ss, const DFVec* __restrict__ uss, const float* __restrict__ As, const float* __restrict__ Bs) {
        constexpr int NQV = NQ / DFV;
        if constexpr (G == 0) {
            const DFVec x0 = xs[0 * NQV];
            const DFVec ux0 = uxs[0 * NQV];
            const DFVec x1 = xs[1 * NQV];
            const DFVec ux1 = uxs[1 * NQV];
            const DFVec x2 = xs[2 * NQV];
            const DFVec ux2 = uxs[2 * NQV];
            const DFVec x3 = xs[3 * NQV];
            const DFVec ux3 = uxs[3 * NQV];
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
            const DFVec sx1_1 = pmul(s1, x1);
            DFVec sxu1_1 = pmul(s1, ux1); pfma(sxu1_1, us1, x1);
            const DFVec sx1_2 = pmul(s1, x2);
            DFVec sxu1_2 = pmul(s1, ux2); pfma(sxu1_2, us1, x2);
            const DFVec sx1_3 = pmul(s1, x3);
            DFVec sxu1_3 = pmul(s1, ux3); pfma(sxu1_3, us1, x3);
            pfma(acc[1], a0.y, sxu1_1);
            pfma(acc[1], b0.y, sx1_1);
            pfma(acc[1], a0.z, sxu1_2);
            pfma(acc[1], b0.z, sx1_2);
            pfma(acc[1], a0.w, sxu1_3);
            pfma(acc[1], b0.w, sx1_3);
            const DFVec s2 = ss[2 * NQV];
            const DFVec us2 = uss[2 * NQV];
            const DFVec sx2_0 = pmul(s2, x0);
            DFVec sxu2_0 = pmul(s2, ux0); pfma(sxu2_0, us2, x0);
            const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
            const float4 b1 = *reinterpret_cast<const float4*>(Bs + 4);
            pfma(acc[2], a1.x, sxu2_0);
            pfma(acc[2], b1.x, sx2_0);
            pfma(acc[3], a1.y, sxu2_0);
            pfma(acc[3], b1.y, sx2_0);
            pfma(acc[4], a1.z, sxu2_0);
            pfma(acc[4], b1.z, sx2_0);
            const DFVec s3 = ss[3 * NQV];
            const DFVec us3 = uss[3 * NQV];
            const DFVec sx3_1 = pmul(s3, x1);
            DFVec sxu3_1 = pmul(s3, ux1); pfma(sxu3_1, us3, x1);
            const DFVec sx3_2 = pmul(s3, x2);
            DFVec sxu3_2 = pmul(s3, ux2); pfma(sxu3_2, us3, x2);
            const DFVec sx3_3 = pmul(s3, x3);
            DFVec sxu3_3 = pmul(s3, ux3); pfma(sxu3_3, us3, x3);
            pfma(acc[5], a1.w, sxu3_1);
            pfma(acc[5], b1.w, sx3_1);
            const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
            const float4 b2 = *reinterpret_cast<const float4*>(Bs + 8);
            pfma(acc[6], a2.x, sxu3_2);
            pfma(acc[6], b2.x, sx3_2);
            pfma(acc[7], a2.y, sxu3_3);
            pfma(acc[7], b2.y, sx3_3);
            const DFVec s4 = ss[4 * NQV];
            const DFVec us4 = uss[4 * NQV];
            const DFVec sx4_1 = pmul(s4, x1);
            DFVec sxu4_1 = pmul(s4, ux1); pfma(sxu4_1, us4, x1);
            const DFVec sx4_2 = pmul(s4, x2);
            DFVec sxu4_2 = pmul(s4, ux2); pfma(sxu4_2, us4, x2);
            const DFVec sx4_3 = pmul(s4, x3);
            DFVec sxu4_3 = pmul(s4, ux3); pfma(sxu4_3, us4, x3);
            pfma(acc[8], a2.z, sxu4_1);
            pfma(acc[8], b2.z, sx4_1);
            pfma(acc[8], a2.w, sxu4_2);
            pfma(acc[8], b2.w, sx4_2);
            const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
            const float4 b3 = *reinterpret_cast<const float4*>(Bs + 12);
            pfma(acc[8], a3.x, sxu4_3);
            pfma(acc[8], b3.x, sx4_3);
        }
        if constexpr (G == 1) {
            const DFVec x0 = xs[0 * NQV];
            const DFVec ux0 = uxs[0 * NQV];
            const DFVec x1 = xs[1 * NQV];
            const DFVec ux1 = uxs[1 * NQV];
            const DFVec x2 = xs[2 * NQV];
            const DFVec ux2 = uxs[2 * NQV];
            const DFVec x3 = xs[3 * NQV];
            const DFVec ux3 = uxs[3 * NQV];
            const DFVec s4 = ss[4 * NQV];
            const DFVec us4 = uss[4 * NQV];
            const DFVec sx4_1 = pmul(s4, x1);
            DFVec sxu4_1 = pmul(s4, ux1); pfma(sxu4_1, us4, x1);
            const DFVec sx4_2 = pmul(s4, x2);
            DFVec sxu4_2 = pmul(s4, ux2); pfma(sxu4_2, us4, x2);
            const DFVec sx4_3 = pmul(s4, x3);
            DFVec sxu4_3 = pmul(s4, ux3); pfma(sxu4_3, us4, x3);
            const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
            const float4 b4 = *reinterpret_cast<const float4*>(Bs + 16);
            pfma(acc[0], a4.x, sxu4_1);
            pfma(acc[0], b4.x, sx4_1);
            pfma(acc[1], a4.w, sxu4_1);
            pfma(acc[1], b4.w, sx4_1);
            pfma(acc[0], a4.y, sxu4_2);
            pfma(acc[0], b4.y, sx4_2);
            const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
            const float4 b5 = *reinterpret_cast<const float4*>(Bs + 20);
            pfma(acc[1], a5.x, sxu4_2);
            pfma(acc[1], b5.x, sx4_2);
            pfma(acc[0], a4.z, sxu4_3);
            pfma(acc[0], b4.z, sx4_3);
            pfma(acc[1], a5.y, sxu4_3);
            pfma(acc[1], b5.y, sx4_3);
            const DFVec s5 = ss[5 * NQV];
            const DFVec us5 = uss[5 * NQV];
            const DFVec sx5_0 = pmul(s5, x0);
            DFVec sxu5_0 = pmul(s5, ux0); pfma(sxu5_0, us5, x0);
            pfma(acc[2], a5.z, sxu5_0);
            pfma(acc[2], b5.z, sx5_0);
            pfma(acc[3], a5.w, sxu5_0);
            pfma(acc[3], b5.w, sx5_0);
            const float4 a6 = *reinterpret_cast<const float4*>(As + 24);
            const float4 b6 = *reinterpret_cast<const float4*>(Bs + 24);
            pfma(acc[4], a6.x, sxu5_0);
            pfma(acc[4], b6.x, sx5_0);
            pfma(acc[5], a6.y, sxu5_0);
            pfma(acc[5], b6.y, sx5_0);
            pfma(acc[6], a6.z, sxu5_0);
            pfma(acc[6], b6.z, sx5_0);
            const DFVec s6 = ss[6 * NQV];
            const DFVec us6 = uss[6 * NQV];
            const DFVec sx6_1 = pmul(s6, x1);
            DFVec sxu6_1 = pmul(s6, ux1); pfma(sxu6_1, us6, x1);
            const DFVec sx6_2 = pmul(s6, x2);
            DFVec sxu6_2 = pmul(s6, ux2); pfma(sxu6_2, us6, x2);
            const DFVec sx6_3 = pmul(s6, x3);
            DFVec sxu6_3 = pmul(s6, ux3); pfma(sxu6_3, us6, x3);
            pfma(acc[7], a6.w, sxu6_1);
            pfma(acc[7], b6.w, sx6_1);
            const float4 a7 = *reinterpret_cast<const float4*>(As + 28);
            const float4 b7 = *reinterpret_cast<const float4*>(Bs + 28);
            pfma(acc[8], a7.y, sxu6_1);
            pfma(acc[8], b7.y, sx6_1);
            pfma(acc[9], a7.w, sxu6_1);
            pfma(acc[9], b7.w, sx6_1);
            const float4 a8 = *reinterpret_cast<const float4*>(As + 32);
            const float4 b8 = *reinterpret_cast<const float4*>(Bs + 32);
            pfma(acc[10], a8.z, sxu6_2);
            pfma(acc[10], b8.z, sx6_2);
            pfma(acc[7], a7.x, sxu6_3);
            pfma(acc[7], b7.x, sx6_3);
            pfma(acc[8], a7.z, sxu6_2);
            pfma(acc[8], b7.z, sx6_2);
            pfma(acc[9], a8.x, sxu6_2);
            pfma(acc[9], b8.x, sx6_2);
            pfma(acc[10], a8.w, sxu6_3);
            pfma(acc[10], b8.w, sx6_3);
            pfma(acc[9], a8.y, sxu6_3);
            pfma(acc[9], b8.y, sx6_3);
        }
        if constexpr (G == 2) {
            const DFVec x0 = xs[0 * NQV];
            const DFVec ux0 = uxs[0 * NQV];
            const DFVec x1 = xs[1 * NQV];
            const DFVec ux1 = uxs[1 * NQV];
            const DFVec x2 = xs[2 * NQV];
            const DFVec ux2 = uxs[2 * NQV];
            const DFVec x3 = xs[3 * NQV];
            const DFVec ux3 = uxs[3 * NQV];
            const DFVec s6 = ss[6 * NQV];
            const DFVec us6 = uss[6 * NQV];
            const DFVec sx6_1 = pmul(s6, x1);
            DFVec sxu6_1 = pmul(s6, ux1); pfma(sxu6_1, us6, x1);
            const DFVec sx6_3 = pmul(s6, x3);
            DFVec sxu6_3 = pmul(s6, ux3); pfma(sxu6_3, us6, x3);
            const float4 a9 = *reinterpret_cast<const float4*>(As + 36);
            const float4 b9 = *reinterpret_cast<const float4*>(Bs + 36);
            pfma(acc[0], a9.x, sxu6_1);
            pfma(acc[0], b9.x, sx6_1);
            pfma(acc[0], a9.y, sxu6_3);
            pfma(acc[0], b9.y, sx6_3);
            const DFVec s7 = ss[7 * NQV];
            const DFVec us7 = uss[7 * NQV];
            const DFVec sx7_1 = pmul(s7, x1);
            DFVec sxu7_1 = pmul(s7, ux1); pfma(sxu7_1, us7, x1);
            const DFVec sx7_2 = pmul(s7, x2);
            DFVec sxu7_2 = pmul(s7, ux2); pfma(sxu7_2, us7, x2);
            const DFVec sx7_3 = pmul(s7, x3);
            DFVec sxu7_3 = pmul(s7, ux3); pfma(sxu7_3, us7, x3);
            pfma(acc[1], a9.z, sxu7_1);
            pfma(acc[1], b9.z, sx7_1);
            const float4 a10 = *reinterpret_cast<const float4*>(As + 40);
            const float4 b10 = *reinterpret_cast<const float4*>(Bs + 40);
            pfma(acc[2], a10.y, sxu7_1);
            pfma(acc[2], b10.y, sx7_1);
            const float4 a11 = *reinterpret_cast<const float4*>(As + 44);
            const float4 b11 = *reinterpret_cast<const float4*>(Bs + 44);
            pfma(acc[3], a11.x, sxu7_1);
            pfma(acc[3], b11.x, sx7_1);
            pfma(acc[4], a11.w, sxu7_1);
            pfma(acc[4], b11.w, sx7_1);
            const float4 a12 = *reinterpret_cast<const float4*>(As + 48);
            const float4 b12 = *reinterpret_cast<const float4*>(Bs + 48);
            pfma(acc[5], a12.z, sxu7_1);
            pfma(acc[5], b12.z, sx7_1);
            pfma(acc[1], a9.w, sxu7_2);
            pfma(acc[1], b9.w, sx7_2);
            pfma(acc[2], a10.z, sxu7_2);
            pfma(acc[2], b10.z, sx7_2);
            pfma(acc[3], a11.y, sxu7_2);
            pfma(acc[3], b11.y, sx7_2);
            pfma(acc[4], a12.x, sxu7_2);
            pfma(acc[4], b12.x, sx7_2);
            pfma(acc[5], a12.w, sxu7_2);
            pfma(acc[5], b12.w, sx7_2);
            pfma(acc[1], a10.x, sxu7_3);
            pfma(acc[1], b10.x, sx7_3);
            pfma(acc[2], a10.w, sxu7_3);
            pfma(acc[2], b10.w, sx7_3);
            pfma(acc[3], a11.z, sxu7_3);
            pfma(acc[3], b11.z, sx7_3);
            pfma(acc[4], a12.y, sxu7_3);
            pfma(acc[4], b12.y, sx7_3);
            const float4 a13 = *reinterpret_cast<const float4*>(As + 52);
            const float4 b13 = *reinterpret_cast<const float4*>(Bs + 52);
            pfma(acc[5], a13.x, sxu7_3);
            pfma(acc[5], b13.x, sx7_3);
            const DFVec s8 = ss[8 * NQV];
            const DFVec us8 = uss[8 * NQV];
            const DFVec sx8_0 = pmul(s8, x0);
            DFVec sxu8_0 = pmul(s8, ux0); pfma(sxu8_0, us8, x0);
            pfma(acc[6], a13.y, sxu8_0);
            pfma(acc[6], b13.y, sx8_0);
            pfma(acc[7], a13.z, sxu8_0);
            pfma(acc[7], b13.z, sx8_0);
            pfma(acc[8], a13.w, sxu8_0);
            pfma(acc[8], b13.w, sx8_0);
            const float4 a14 = *reinterpret_cast<const float4*>(As + 56);
            const float4 b14 = *reinterpret_cast<const float4*>(Bs + 56);
            pfma(acc[9], a14.x, sxu8_0);
            pfma(acc[9], b14.x, sx8_0);
        }
        if constexpr (G == 3) {
            const DFVec x0 = xs[0 * NQV];
            const DFVec ux0 = uxs[0 * NQV];
            const DFVec x1 = xs[1 * NQV];
            const DFVec ux1 = uxs[1 * NQV];
            const DFVec x2 = xs[2 * NQV];
            const DFVec ux2 = uxs[2 * NQV];
            const DFVec x3 = xs[3 * NQV];
            const DFVec ux3 = uxs[3 * NQV];
            const DFVec s8 = ss[8 * NQV];
            const DFVec us8 = uss[8 * NQV];
            const DFVec sx8_0 = pmul(s8, x0);
            DFVec sxu8_0 = pmul(s8, ux0); pfma(sxu8_0, us8, x0);
            const float4 a15 = *reinterpret_cast<const float4*>(As + 60);
            const float4 b15 = *reinterpret_cast<const float4*>(Bs + 60);
            pfma(acc[0], a15.x, sxu8_0);
            pfma(acc[0], b15.x, sx8_0);
            pfma(acc[1], a15.y, sxu8_0);
            pfma(acc[1], b15.y, sx8_0);
            pfma(acc[2], a15.z, sxu8_0);
            pfma(acc[2], b15.z, sx8_0);
            const DFVec s9 = ss[9 * NQV];
            const DFVec us9 = uss[9 * NQV];
            const DFVec sx9_1 = pmul(s9, x1);
            DFVec sxu9_1 = pmul(s9, ux1); pfma(sxu9_1, us9, x1);
            const DFVec sx9_2 = pmul(s9, x2);
            DFVec sxu9_2 = pmul(s9, ux2); pfma(sxu9_2, us9, x2);
            const DFVec sx9_3 = pmul(s9, x3);
            DFVec sxu9_3 = pmul(s9, ux3); pfma(sxu9_3, us9, x3);
            pfma(acc[3], a15.w, sxu9_1);
            pfma(acc[3], b15.w, sx9_1);
            const float4 a16 = *reinterpret_cast<const float4*>(As + 64);
            const float4 b16 = *reinterpret_cast<const float4*>(Bs + 64);
            pfma(acc[4], a16.y, sxu9_1);
            pfma(acc[4], b16.y, sx9_1);
            const float4 a17 = *reinterpret_cast<const float4*>(As + 68);
            const float4 b17 = *reinterpret_cast<const float4*>(Bs + 68);
            pfma(acc[5], a17.x, sxu9_1);
            pfma(acc[5], b17.x, sx9_1);
            pfma(acc[6], a17.w, sxu9_1);
            pfma(acc[6], b17.w, sx9_1);
            const float4 a18 = *reinterpret_cast<const float4*>(As + 72);
            const float4 b18 = *reinterpret_cast<const float4*>(Bs + 72);
            pfma(acc[7], a18.z, sxu9_1);
            pfma(acc[7], b18.z, sx9_1);
            const float4 a19 = *reinterpret_cast<const float4*>(As + 76);
            const float4 b19 = *reinterpret_cast<const float4*>(Bs + 76);
            pfma(acc[8], a19.y, sxu9_1);
            pfma(acc[8], b19.y, sx9_1);
            const float4 a20 = *reinterpret_cast<const float4*>(As + 80);
            const float4 b20 = *reinterpret_cast<const float4*>(Bs + 80);
            pfma(acc[9], a20.x, sxu9_1);
            pfma(acc[9], b20.x, sx9_1);
            pfma(acc[3], a16.x, sxu9_3);
            pfma(acc[3], b16.x, sx9_3);
            pfma(acc[4], a16.z, sxu9_2);
            pfma(acc[4], b16.z, sx9_2);
            pfma(acc[5], a17.y, sxu9_2);
            pfma(acc[5], b17.y, sx9_2);
            pfma(acc[6], a18.x, sxu9_2);
            pfma(acc[6], b18.x, sx9_2);
            pfma(acc[7], a18.w, sxu9_2);
            pfma(acc[7], b18.w, sx9_2);
            pfma(acc[8], a19.z, sxu9_2);
            pfma(acc[8], b19.z, sx9_2);
            pfma(acc[9], a20.y, sxu9_3);
            pfma(acc[9], b20.y, sx9_3);
            pfma(acc[4], a16.w, sxu9_3);
            pfma(acc[4], b16.w, sx9_3);
            pfma(acc[5], a17.z, sxu9_3);
            pfma(acc[5], b17.z, sx9_3);
            pfma(acc[6], a18.y, sxu9_3);
            pfma(acc[6], b18.y, sx9_3);
            pfma(acc[7], a19.x, sxu9_3);
            pfma(acc[7], b19.x, sx9_3);
            pfma(acc[8], a19.w, sxu9_3);
            pfma(acc[8], b19.w, sx9_3);
        }
    }
    // writes the group's rows to dst[r * stride] (dst already offset by the lane and the first row)
    template <int G, class VecT>
    __device__ static __forceinline__ void fwd_store(const VecT (&acc)[F_RMAX], VecT* __restrict__ dst, const int stride) {
        if constexpr (G == 0) {
            dst[0 * stride] = acc[0];
            dst[1 * stride] = acc[1];
            dst[2 * stride] = acc[2];
            dst[3 * stride] = acc[3];
            dst[4 * stride] = acc[4];
            dst[5 * stride] = acc[5];
            dst[6 * stride] = acc[6];
            dst[7 * stride] = acc[7];
            dst[8 * stride] = acc[8];
        }
        if constexpr (G == 1) {
            dst[0 * stride] = acc[0];
            dst[1 * stride] = acc[1];
            dst[2 * stride] = acc[2];
            dst[3 * stride] = acc[3];
            dst[4 * stride] = acc[4];
            dst[5 * stride] = acc[5];
            dst[6 * stride] = acc[6];
            dst[7 * stride] = acc[7];
            dst[8 * stride] = acc[8];
            dst[9 * stride] = acc[9];
            dst[10 * stride] = acc[10];
        }
        if constexpr (G == 2) {
            dst[0 * stride] = acc[0];
            dst[1 * stride] = acc[1];
            dst[2 * stride] = acc[2];
            dst[3 * stride] = acc[3];
            dst[4 * stride] = acc[4];
            dst[5 * stride] = acc[5];
            dst[6 * stride] = acc[6];
            dst[7 * stride] = acc[7];
            dst[8 * stride] = acc[8];
            dst[9 * stride] = acc[9];
        }
        if constexpr (G == 3) {
            dst[0 * stride] = acc[0];
            dst[1 * stride] = acc[1];
            dst[2 * stride] = acc[2];
            dst[3 * stride] = acc[3];
            dst[4 * stride] = acc[4];
            dst[5 * stride] = acc[5];
            dst[6 * stride] = acc[6];
            dst[7 * stride] = acc[7];
            dst[8 * stride] = acc[8];
            dst[9 * stride] = acc[9];
        }
    }
    // ---- backward: path groups [[0, 5, 6], [1, 3, 4], [2, 9], [7, 8]]
    static constexpr int BV = 4;  // channels per lane in the backward
    using BVec = float4;
    static constexpr int BW = 4, BT = 5, BS = 2, BC = 2, B_RMAX = 12, B_APAD = 84, B_NREC = 2;
    // edge-wise backward (one warp per edge, grad_out rows read from shared memory): edges per tile (0 = not generated), ring stages
    static constexpr int ET = 11, ES = 2, EV = 4, EXG = 0;   // EXG: sender rows not staged
    static constexpr int ST = 11;   // columns of the scheduled backward
    // the same for the standalone tensor product: rows per ring slot (0 = not generated), ring slots
    static constexpr int ETR = 0, ESR = 3;
    // fused double backward (edge outputs): edges per tile (0 = not generated), ring stages
    static constexpr int DT = 4, DS = 2, DV = 2;
    using DVec = float2;
    using EVec = float4;
    __device__ static __forceinline__ PairRec b_pair_rec(int i) { return kBPair_w128_l3_natural[i]; }
    __device__ static __forceinline__ float b_rec_val(int i) { return kBVal_w128_l3_natural[i]; }
    __device__ static __forceinline__ unsigned char b_rec_i2(int i) { return kBI2_w128_l3_natural[i]; }
    // output rows of path group g: b_nrow(g) of them, the r-th is b_row(g, r)
    __device__ static __forceinline__ int b_row(int g, int r) { return kBRow_w128_l3_natural[g * B_RMAX + r]; }
    static constexpr int b_nrow(int g) {
        switch (g) {
            case 0: return 11;
            case 1: return 7;
            case 2: return 10;
            case 3: return 12;
            default: return 0;
        }
    }
    __device__ static __forceinline__ void bwd_edge(const int G, const BVec (&dm)[B_RMAX], const BVec* __restrict__ xs, const BVec* __restrict__ ss, const float* __restrict__ As, BVec (&dxp)[DIN], float (&dyl)[16], BVec* __restrict__ gw) {
        constexpr int NQV = NQ / BV;
        switch (G) {
        case 0: {
            const BVec x0 = xs[0 * NQV];
            const BVec x1 = xs[1 * NQV];
            const BVec x2 = xs[2 * NQV];
            const BVec x3 = xs[3 * NQV];
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
            const BVec s5 = ss[5 * NQV];  // path 5: l1=0 l2=2 -> L=2
            const BVec sx5_0 = vmul(s5, x0);
            BVec u5_0; vzero(u5_0);
            vfma(u5_0, a0.y, dm[1]);
            { const float t = vdot(sx5_0, dm[1]);
              dyl[4] = 1.0f * t;
            }
            vfma(u5_0, a0.z, dm[2]);
            { const float t = vdot(sx5_0, dm[2]);
              dyl[5] = 1.0f * t;
            }
            vfma(u5_0, a0.w, dm[3]);
            { const float t = vdot(sx5_0, dm[3]);
              dyl[6] = 1.0f * t;
            }
            const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
            vfma(u5_0, a1.x, dm[4]);
            { const float t = vdot(sx5_0, dm[4]);
              dyl[7] = 1.0f * t;
            }
            vfma(u5_0, a1.y, dm[5]);
            { const float t = vdot(sx5_0, dm[5]);
              dyl[8] = 1.0f * t;
            }
            BVec ds5 = vmul(x0, u5_0);
            if (gw) gw[5 * NQV] = ds5;
            vfma(dxp[0], s5, u5_0);
            const BVec s6 = ss[6 * NQV];  // path 6: l1=1 l2=1 -> L=2
            const BVec sx6_1 = vmul(s6, x1);
            BVec u6_1; vzero(u6_1);
            const BVec sx6_2 = vmul(s6, x2);
            BVec u6_2; vzero(u6_2);
            const BVec sx6_3 = vmul(s6, x3);
            BVec u6_3; vzero(u6_3);
            vfma(u6_1, a1.z, dm[6]);
            { const float t = vdot(sx6_1, dm[6]);
              dyl[3] = 0.707106769f * t;
            }
            const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
            vfma(u6_1, a2.x, dm[7]);
            { const float t = vdot(sx6_1, dm[7]);
              dyl[2] = 0.707106769f * t;
            }
            vfma(u6_1, a2.z, dm[8]);
            { const float t = vdot(sx6_1, dm[8]);
              dyl[1] = -0.408248305f * t;
            }
            const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
            vfma(u6_2, a3.y, dm[9]);
            { const float t = vdot(sx6_2, dm[9]);
              dyl[3] = fmaf(0.707106769f, t, dyl[3]);
            }
            vfma(u6_1, a3.w, dm[10]);
            { const float t = vdot(sx6_1, dm[10]);
              dyl[1] = fmaf(-0.707106769f, t, dyl[1]);
            }
            vfma(u6_3, a1.w, dm[6]);
            { const float t = vdot(sx6_3, dm[6]);
              dyl[1] = fmaf(0.707106769f, t, dyl[1]);
            }
            vfma(u6_2, a2.y, dm[7]);
            { const float t = vdot(sx6_2, dm[7]);
              dyl[1] = fmaf(0.707106769f, t, dyl[1]);
            }
            vfma(u6_2, a2.w, dm[8]);
            { const float t = vdot(sx6_2, dm[8]);
              dyl[2] = fmaf(0.816496611f, t, dyl[2]);
            }
            vfma(u6_3, a3.z, dm[9]);
            { const float t = vdot(sx6_3, dm[9]);
              dyl[2] = fmaf(0.707106769f, t, dyl[2]);
            }
            const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
            vfma(u6_3, a4.x, dm[10]);
            { const float t = vdot(sx6_3, dm[10]);
              dyl[3] = fmaf(0.707106769f, t, dyl[3]);
            }
            vfma(u6_3, a3.x, dm[8]);
            { const float t = vdot(sx6_3, dm[8]);
              dyl[3] = fmaf(-0.408248305f, t, dyl[3]);
            }
            BVec ds6 = vmul(x1, u6_1);
            vfma(ds6, x2, u6_2);
            vfma(ds6, x3, u6_3);
            if (gw) gw[6 * NQV] = ds6;
            dxp[1] = vmul(s6, u6_1);
            dxp[2] = vmul(s6, u6_2);
            dxp[3] = vmul(s6, u6_3);
            dyl[9] = 0.f;
            dyl[10] = 0.f;
            dyl[11] = 0.f;
            dyl[12] = 0.f;
            dyl[13] = 0.f;
            dyl[14] = 0.f;
            dyl[15] = 0.f;
        } break;
        case 1: {
            const BVec x1 = xs[1 * NQV];
            const BVec x2 = xs[2 * NQV];
            const BVec x3 = xs[3 * NQV];
            const BVec s1 = ss[1 * NQV];  // path 1: l1=1 l2=1 -> L=0
            const BVec sx1_1 = vmul(s1, x1);
            BVec u1_1; vzero(u1_1);
            const BVec sx1_2 = vmul(s1, x2);
            BVec u1_2; vzero(u1_2);
            const BVec sx1_3 = vmul(s1, x3);
            BVec u1_3; vzero(u1_3);
            const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
            vfma(u1_1, a5.x, dm[0]);
            { const float t = vdot(sx1_1, dm[0]);
              dyl[1] = 0.577350259f * t;
            }
            vfma(u1_2, a5.y, dm[0]);
            { const float t = vdot(sx1_2, dm[0]);
              dyl[2] = 0.577350259f * t;
            }
            vfma(u1_3, a5.z, dm[0]);
            { const float t = vdot(sx1_3, dm[0]);
              dyl[3] = 0.577350259f * t;
            }
            BVec ds1 = vmul(x1, u1_1);
            vfma(ds1, x2, u1_2);
            vfma(ds1, x3, u1_3);
            if (gw) gw[1 * NQV] = ds1;
            dxp[1] = vmul(s1, u1_1);
            dxp[2] = vmul(s1, u1_2);
            dxp[3] = vmul(s1, u1_3);
            const BVec s3 = ss[3 * NQV];  // path 3: l1=1 l2=0 -> L=1
            const BVec sx3_1 = vmul(s3, x1);
            BVec u3_1; vzero(u3_1);
            const BVec sx3_2 = vmul(s3, x2);
            BVec u3_2; vzero(u3_2);
            const BVec sx3_3 = vmul(s3, x3);
            BVec u3_3; vzero(u3_3);
            vfma(u3_1, a5.w, dm[1]);
            { const float t = vdot(sx3_1, dm[1]);
              dyl[0] = 1.0f * t;
            }
            const float4 a6 = *reinterpret_cast<const float4*>(As + 24);
            vfma(u3_2, a6.x, dm[2]);
            { const float t = vdot(sx3_2, dm[2]);
              dyl[0] = fmaf(1.0f, t, dyl[0]);
            }
            vfma(u3_3, a6.y, dm[3]);
            { const float t = vdot(sx3_3, dm[3]);
              dyl[0] = fmaf(1.0f, t, dyl[0]);
            }
            BVec ds3 = vmul(x1, u3_1);
            vfma(ds3, x2, u3_2);
            vfma(ds3, x3, u3_3);
            if (gw) gw[3 * NQV] = ds3;
            vfma(dxp[1], s3, u3_1);
            vfma(dxp[2], s3, u3_2);
            vfma(dxp[3], s3, u3_3);
            const BVec s4 = ss[4 * NQV];  // path 4: l1=1 l2=2 -> L=1
            const BVec sx4_1 = vmul(s4, x1);
            BVec u4_1; vzero(u4_1);
            const BVec sx4_2 = vmul(s4, x2);
            BVec u4_2; vzero(u4_2);
            const BVec sx4_3 = vmul(s4, x3);
            BVec u4_3; vzero(u4_3);
            vfma(u4_1, a6.z, dm[4]);
            { const float t = vdot(sx4_1, dm[4]);
              dyl[6] = 0.316227764f * t;
              dyl[8] = 0.547722578f * t;
            }
            const float4 a7 = *reinterpret_cast<const float4*>(As + 28);
            vfma(u4_1, a7.y, dm[5]);
            { const float t = vdot(sx4_1, dm[5]);
              dyl[5] = -0.547722578f * t;
            }
            const float4 a8 = *reinterpret_cast<const float4*>(As + 32);
            vfma(u4_1, a8.x, dm[6]);
            { const float t = vdot(sx4_1, dm[6]);
              dyl[4] = -0.547722578f * t;
            }
            vfma(u4_2, a6.w, dm[4]);
            { const float t = vdot(sx4_2, dm[4]);
              dyl[5] = fmaf(-0.547722578f, t, dyl[5]);
            }
            vfma(u4_2, a7.z, dm[5]);
            { const float t = vdot(sx4_2, dm[5]);
              dyl[6] = fmaf(-0.632455528f, t, dyl[6]);
            }
            vfma(u4_2, a8.y, dm[6]);
            { const float t = vdot(sx4_2, dm[6]);
              dyl[7] = -0.547722578f * t;
            }
            vfma(u4_3, a7.x, dm[4]);
            { const float t = vdot(sx4_3, dm[4]);
              dyl[4] = fmaf(-0.547722578f, t, dyl[4]);
            }
            vfma(u4_3, a7.w, dm[5]);
            { const float t = vdot(sx4_3, dm[5]);
              dyl[7] = fmaf(-0.547722578f, t, dyl[7]);
            }
            vfma(u4_3, a8.z, dm[6]);
            { const float t = vdot(sx4_3, dm[6]);
              dyl[6] = fmaf(0.316227764f, t, dyl[6]);
              dyl[8] = fmaf(-0.547722578f, t, dyl[8]);
            }
            BVec ds4 = vmul(x1, u4_1);
            vfma(ds4, x2, u4_2);
            vfma(ds4, x3, u4_3);
            if (gw) gw[4 * NQV] = ds4;
            vfma(dxp[1], s4, u4_1);
            vfma(dxp[2], s4, u4_2);
            vfma(dxp[3], s4, u4_3);
            vzero(dxp[0]);
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
            const BVec x1 = xs[1 * NQV];
            const BVec x2 = xs[2 * NQV];
            const BVec x3 = xs[3 * NQV];
            const BVec s2 = ss[2 * NQV];  // path 2: l1=0 l2=1 -> L=1
            const BVec sx2_0 = vmul(s2, x0);
            BVec u2_0; vzero(u2_0);
            const float4 a9 = *reinterpret_cast<const float4*>(As + 36);
            vfma(u2_0, a9.x, dm[0]);
            { const float t = vdot(sx2_0, dm[0]);
              dyl[1] = 1.0f * t;
            }
            vfma(u2_0, a9.y, dm[1]);
            { const float t = vdot(sx2_0, dm[1]);
              dyl[2] = 1.0f * t;
            }
            vfma(u2_0, a9.z, dm[2]);
            { const float t = vdot(sx2_0, dm[2]);
              dyl[3] = 1.0f * t;
            }
            BVec ds2 = vmul(x0, u2_0);
            if (gw) gw[2 * NQV] = ds2;
            dxp[0] = vmul(s2, u2_0);
            const BVec s9 = ss[9 * NQV];  // path 9: l1=1 l2=2 -> L=3
            const BVec sx9_1 = vmul(s9, x1);
            BVec u9_1; vzero(u9_1);
            const BVec sx9_2 = vmul(s9, x2);
            BVec u9_2; vzero(u9_2);
            const BVec sx9_3 = vmul(s9, x3);
            BVec u9_3; vzero(u9_3);
            vfma(u9_1, a9.w, dm[3]);
            { const float t = vdot(sx9_1, dm[3]);
              dyl[8] = 0.707106769f * t;
            }
            const float4 a10 = *reinterpret_cast<const float4*>(As + 40);
            vfma(u9_1, a10.y, dm[4]);
            { const float t = vdot(sx9_1, dm[4]);
              dyl[7] = 0.577350259f * t;
            }
            const float4 a11 = *reinterpret_cast<const float4*>(As + 44);
            vfma(u9_1, a11.x, dm[5]);
            { const float t = vdot(sx9_1, dm[5]);
              dyl[6] = 0.632455528f * t;
              dyl[8] = fmaf(0.182574183f, t, dyl[8]);
            }
            vfma(u9_1, a11.w, dm[6]);
            { const float t = vdot(sx9_1, dm[6]);
              dyl[5] = -0.44721359f * t;
            }
            const float4 a12 = *reinterpret_cast<const float4*>(As + 48);
            vfma(u9_1, a12.z, dm[7]);
            { const float t = vdot(sx9_1, dm[7]);
              dyl[4] = -0.182574183f * t;
            }
            const float4 a13 = *reinterpret_cast<const float4*>(As + 52);
            vfma(u9_1, a13.y, dm[8]);
            { const float t = vdot(sx9_1, dm[8]);
              dyl[5] = fmaf(-0.577350259f, t, dyl[5]);
            }
            const float4 a14 = *reinterpret_cast<const float4*>(As + 56);
            vfma(u9_1, a14.x, dm[9]);
            { const float t = vdot(sx9_1, dm[9]);
              dyl[4] = fmaf(-0.707106769f, t, dyl[4]);
            }
            vfma(u9_3, a10.x, dm[3]);
            { const float t = vdot(sx9_3, dm[3]);
              dyl[4] = fmaf(0.707106769f, t, dyl[4]);
            }
            vfma(u9_2, a10.z, dm[4]);
            { const float t = vdot(sx9_2, dm[4]);
              dyl[4] = fmaf(0.577350259f, t, dyl[4]);
            }
            vfma(u9_2, a11.y, dm[5]);
            { const float t = vdot(sx9_2, dm[5]);
              dyl[5] = fmaf(0.730296731f, t, dyl[5]);
            }
            vfma(u9_2, a12.x, dm[6]);
            { const float t = vdot(sx9_2, dm[6]);
              dyl[6] = fmaf(0.774596691f, t, dyl[6]);
            }
            vfma(u9_2, a12.w, dm[7]);
            { const float t = vdot(sx9_2, dm[7]);
              dyl[7] = fmaf(0.730296731f, t, dyl[7]);
            }
            vfma(u9_2, a13.z, dm[8]);
            { const float t = vdot(sx9_2, dm[8]);
              dyl[8] = fmaf(0.577350259f, t, dyl[8]);
            }
            vfma(u9_3, a14.y, dm[9]);
            { const float t = vdot(sx9_3, dm[9]);
              dyl[8] = fmaf(0.707106769f, t, dyl[8]);
            }
            vfma(u9_3, a10.w, dm[4]);
            { const float t = vdot(sx9_3, dm[4]);
              dyl[5] = fmaf(0.577350259f, t, dyl[5]);
            }
            vfma(u9_3, a11.z, dm[5]);
            { const float t = vdot(sx9_3, dm[5]);
              dyl[4] = fmaf(-0.182574183f, t, dyl[4]);
            }
            vfma(u9_3, a12.y, dm[6]);
            { const float t = vdot(sx9_3, dm[6]);
              dyl[7] = fmaf(-0.44721359f, t, dyl[7]);
            }
            vfma(u9_3, a13.x, dm[7]);
            { const float t = vdot(sx9_3, dm[7]);
              dyl[6] = fmaf(0.632455528f, t, dyl[6]);
              dyl[8] = fmaf(-0.182574183f, t, dyl[8]);
            }
            vfma(u9_3, a13.w, dm[8]);
            { const float t = vdot(sx9_3, dm[8]);
              dyl[7] = fmaf(0.577350259f, t, dyl[7]);
            }
            BVec ds9 = vmul(x1, u9_1);
            vfma(ds9, x2, u9_2);
            vfma(ds9, x3, u9_3);
            if (gw) gw[9 * NQV] = ds9;
            dxp[1] = vmul(s9, u9_1);
            dxp[2] = vmul(s9, u9_2);
            dxp[3] = vmul(s9, u9_3);
            dyl[0] = 0.f;
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
            const BVec x1 = xs[1 * NQV];
            const BVec x2 = xs[2 * NQV];
            const BVec x3 = xs[3 * NQV];
            const BVec s7 = ss[7 * NQV];  // path 7: l1=1 l2=3 -> L=2
            const BVec sx7_1 = vmul(s7, x1);
            BVec u7_1; vzero(u7_1);
            const BVec sx7_2 = vmul(s7, x2);
            BVec u7_2; vzero(u7_2);
            const BVec sx7_3 = vmul(s7, x3);
            BVec u7_3; vzero(u7_3);
            const float4 a15 = *reinterpret_cast<const float4*>(As + 60);
            vfma(u7_1, a15.x, dm[0]);
            { const float t = vdot(sx7_1, dm[0]);
              dyl[13] = 0.154303357f * t;
              dyl[15] = 0.597614288f * t;
            }
            vfma(u7_1, a15.w, dm[1]);
            { const float t = vdot(sx7_1, dm[1]);
              dyl[12] = 0.377964467f * t;
              dyl[14] = 0.487950027f * t;
            }
            const float4 a16 = *reinterpret_cast<const float4*>(As + 64);
            vfma(u7_1, a16.z, dm[2]);
            { const float t = vdot(sx7_1, dm[2]);
              dyl[11] = -0.534522474f * t;
            }
            const float4 a17 = *reinterpret_cast<const float4*>(As + 68);
            vfma(u7_1, a17.y, dm[3]);
            { const float t = vdot(sx7_1, dm[3]);
              dyl[10] = -0.487950027f * t;
            }
            const float4 a18 = *reinterpret_cast<const float4*>(As + 72);
            vfma(u7_1, a18.x, dm[4]);
            { const float t = vdot(sx7_1, dm[4]);
              dyl[9] = -0.597614288f * t;
              dyl[11] = fmaf(-0.154303357f, t, dyl[11]);
            }
            vfma(u7_2, a15.y, dm[0]);
            { const float t = vdot(sx7_2, dm[0]);
              dyl[10] = fmaf(-0.487950027f, t, dyl[10]);
            }
            vfma(u7_2, a16.x, dm[1]);
            { const float t = vdot(sx7_2, dm[1]);
              dyl[11] = fmaf(-0.617213428f, t, dyl[11]);
            }
            vfma(u7_2, a16.w, dm[2]);
            { const float t = vdot(sx7_2, dm[2]);
              dyl[12] = fmaf(-0.654653668f, t, dyl[12]);
            }
            vfma(u7_2, a17.z, dm[3]);
            { const float t = vdot(sx7_2, dm[3]);
              dyl[13] = fmaf(-0.617213428f, t, dyl[13]);
            }
            vfma(u7_2, a18.y, dm[4]);
            { const float t = vdot(sx7_2, dm[4]);
              dyl[14] = fmaf(-0.487950027f, t, dyl[14]);
            }
            vfma(u7_3, a15.z, dm[0]);
            { const float t = vdot(sx7_3, dm[0]);
              dyl[9] = fmaf(-0.597614288f, t, dyl[9]);
              dyl[11] = fmaf(0.154303357f, t, dyl[11]);
            }
            vfma(u7_3, a16.y, dm[1]);
            { const float t = vdot(sx7_3, dm[1]);
              dyl[10] = fmaf(-0.487950027f, t, dyl[10]);
            }
            vfma(u7_3, a17.x, dm[2]);
            { const float t = vdot(sx7_3, dm[2]);
              dyl[13] = fmaf(-0.534522474f, t, dyl[13]);
            }
            vfma(u7_3, a17.w, dm[3]);
            { const float t = vdot(sx7_3, dm[3]);
              dyl[12] = fmaf(0.377964467f, t, dyl[12]);
              dyl[14] = fmaf(-0.487950027f, t, dyl[14]);
            }
            vfma(u7_3, a18.z, dm[4]);
            { const float t = vdot(sx7_3, dm[4]);
              dyl[13] = fmaf(0.154303357f, t, dyl[13]);
              dyl[15] = fmaf(-0.597614288f, t, dyl[15]);
            }
            BVec ds7 = vmul(x1, u7_1);
            vfma(ds7, x2, u7_2);
            vfma(ds7, x3, u7_3);
            if (gw) gw[7 * NQV] = ds7;
            dxp[1] = vmul(s7, u7_1);
            dxp[2] = vmul(s7, u7_2);
            dxp[3] = vmul(s7, u7_3);
            const BVec s8 = ss[8 * NQV];  // path 8: l1=0 l2=3 -> L=3
            const BVec sx8_0 = vmul(s8, x0);
            BVec u8_0; vzero(u8_0);
            vfma(u8_0, a18.w, dm[5]);
            { const float t = vdot(sx8_0, dm[5]);
              dyl[9] = fmaf(1.0f, t, dyl[9]);
            }
            const float4 a19 = *reinterpret_cast<const float4*>(As + 76);
            vfma(u8_0, a19.x, dm[6]);
            { const float t = vdot(sx8_0, dm[6]);
              dyl[10] = fmaf(1.0f, t, dyl[10]);
            }
            vfma(u8_0, a19.y, dm[7]);
            { const float t = vdot(sx8_0, dm[7]);
              dyl[11] = fmaf(1.0f, t, dyl[11]);
            }
            vfma(u8_0, a19.z, dm[8]);
            { const float t = vdot(sx8_0, dm[8]);
              dyl[12] = fmaf(1.0f, t, dyl[12]);
            }
            vfma(u8_0, a19.w, dm[9]);
            { const float t = vdot(sx8_0, dm[9]);
              dyl[13] = fmaf(1.0f, t, dyl[13]);
            }
            const float4 a20 = *reinterpret_cast<const float4*>(As + 80);
            vfma(u8_0, a20.x, dm[10]);
            { const float t = vdot(sx8_0, dm[10]);
              dyl[14] = fmaf(1.0f, t, dyl[14]);
            }
            vfma(u8_0, a20.y, dm[11]);
            { const float t = vdot(sx8_0, dm[11]);
              dyl[15] = fmaf(1.0f, t, dyl[15]);
            }
            BVec ds8 = vmul(x0, u8_0);
            if (gw) gw[8 * NQV] = ds8;
            dxp[0] = vmul(s8, u8_0);
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
        const EVec x1 = xs[1 * NQV];
        const EVec x2 = xs[2 * NQV];
        const EVec x3 = xs[3 * NQV];
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
        const EVec s1 = ss[1 * NQV];  // path 1: l1=1 l2=1 -> L=0
        const EVec sx1_1 = vmul(s1, x1);
        EVec u1_1; vzero(u1_1);
        const EVec sx1_2 = vmul(s1, x2);
        EVec u1_2; vzero(u1_2);
        const EVec sx1_3 = vmul(s1, x3);
        EVec u1_3; vzero(u1_3);
        const EVec d1_1 = dms[1 * NQV];
        const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
        vfma(u1_1, a5.x, d1_1);
        { const float t = vdot(sx1_1, d1_1);
          dyl[1] = 0.577350259f * t;
        }
        vfma(u1_2, a5.y, d1_1);
        { const float t = vdot(sx1_2, d1_1);
          dyl[2] = 0.577350259f * t;
        }
        vfma(u1_3, a5.z, d1_1);
        { const float t = vdot(sx1_3, d1_1);
          dyl[3] = 0.577350259f * t;
        }
        EVec ds1 = vmul(x1, u1_1);
        vfma(ds1, x2, u1_2);
        vfma(ds1, x3, u1_3);
        if (gw) gw[1 * NQV] = ds1;
        dxp[1] = vmul(s1, u1_1);
        dxp[2] = vmul(s1, u1_2);
        dxp[3] = vmul(s1, u1_3);
        const EVec s2 = ss[2 * NQV];  // path 2: l1=0 l2=1 -> L=1
        const EVec sx2_0 = vmul(s2, x0);
        EVec u2_0; vzero(u2_0);
        const EVec d2_2 = dms[2 * NQV];
        const float4 a9 = *reinterpret_cast<const float4*>(As + 36);
        vfma(u2_0, a9.x, d2_2);
        { const float t = vdot(sx2_0, d2_2);
          dyl[1] = fmaf(1.0f, t, dyl[1]);
        }
        const EVec d2_3 = dms[3 * NQV];
        vfma(u2_0, a9.y, d2_3);
        { const float t = vdot(sx2_0, d2_3);
          dyl[2] = fmaf(1.0f, t, dyl[2]);
        }
        const EVec d2_4 = dms[4 * NQV];
        vfma(u2_0, a9.z, d2_4);
        { const float t = vdot(sx2_0, d2_4);
          dyl[3] = fmaf(1.0f, t, dyl[3]);
        }
        EVec ds2 = vmul(x0, u2_0);
        if (gw) gw[2 * NQV] = ds2;
        vfma(dxp[0], s2, u2_0);
        const EVec s3 = ss[3 * NQV];  // path 3: l1=1 l2=0 -> L=1
        const EVec sx3_1 = vmul(s3, x1);
        EVec u3_1; vzero(u3_1);
        const EVec sx3_2 = vmul(s3, x2);
        EVec u3_2; vzero(u3_2);
        const EVec sx3_3 = vmul(s3, x3);
        EVec u3_3; vzero(u3_3);
        const EVec d3_5 = dms[5 * NQV];
        vfma(u3_1, a5.w, d3_5);
        { const float t = vdot(sx3_1, d3_5);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        const EVec d3_6 = dms[6 * NQV];
        const float4 a6 = *reinterpret_cast<const float4*>(As + 24);
        vfma(u3_2, a6.x, d3_6);
        { const float t = vdot(sx3_2, d3_6);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        const EVec d3_7 = dms[7 * NQV];
        vfma(u3_3, a6.y, d3_7);
        { const float t = vdot(sx3_3, d3_7);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        EVec ds3 = vmul(x1, u3_1);
        vfma(ds3, x2, u3_2);
        vfma(ds3, x3, u3_3);
        if (gw) gw[3 * NQV] = ds3;
        vfma(dxp[1], s3, u3_1);
        vfma(dxp[2], s3, u3_2);
        vfma(dxp[3], s3, u3_3);
        const EVec s4 = ss[4 * NQV];  // path 4: l1=1 l2=2 -> L=1
        const EVec sx4_1 = vmul(s4, x1);
        EVec u4_1; vzero(u4_1);
        const EVec sx4_2 = vmul(s4, x2);
        EVec u4_2; vzero(u4_2);
        const EVec sx4_3 = vmul(s4, x3);
        EVec u4_3; vzero(u4_3);
        const EVec d4_8 = dms[8 * NQV];
        vfma(u4_1, a6.z, d4_8);
        { const float t = vdot(sx4_1, d4_8);
          dyl[6] = 0.316227764f * t;
          dyl[8] = 0.547722578f * t;
        }
        const EVec d4_9 = dms[9 * NQV];
        const float4 a7 = *reinterpret_cast<const float4*>(As + 28);
        vfma(u4_1, a7.y, d4_9);
        { const float t = vdot(sx4_1, d4_9);
          dyl[5] = -0.547722578f * t;
        }
        const EVec d4_10 = dms[10 * NQV];
        const float4 a8 = *reinterpret_cast<const float4*>(As + 32);
        vfma(u4_1, a8.x, d4_10);
        { const float t = vdot(sx4_1, d4_10);
          dyl[4] = -0.547722578f * t;
        }
        vfma(u4_2, a6.w, d4_8);
        { const float t = vdot(sx4_2, d4_8);
          dyl[5] = fmaf(-0.547722578f, t, dyl[5]);
        }
        vfma(u4_2, a7.z, d4_9);
        { const float t = vdot(sx4_2, d4_9);
          dyl[6] = fmaf(-0.632455528f, t, dyl[6]);
        }
        vfma(u4_2, a8.y, d4_10);
        { const float t = vdot(sx4_2, d4_10);
          dyl[7] = -0.547722578f * t;
        }
        vfma(u4_3, a7.x, d4_8);
        { const float t = vdot(sx4_3, d4_8);
          dyl[4] = fmaf(-0.547722578f, t, dyl[4]);
        }
        vfma(u4_3, a7.w, d4_9);
        { const float t = vdot(sx4_3, d4_9);
          dyl[7] = fmaf(-0.547722578f, t, dyl[7]);
        }
        vfma(u4_3, a8.z, d4_10);
        { const float t = vdot(sx4_3, d4_10);
          dyl[6] = fmaf(0.316227764f, t, dyl[6]);
          dyl[8] = fmaf(-0.547722578f, t, dyl[8]);
        }
        EVec ds4 = vmul(x1, u4_1);
        vfma(ds4, x2, u4_2);
        vfma(ds4, x3, u4_3);
        if (gw) gw[4 * NQV] = ds4;
        vfma(dxp[1], s4, u4_1);
        vfma(dxp[2], s4, u4_2);
        vfma(dxp[3], s4, u4_3);
        const EVec s5 = ss[5 * NQV];  // path 5: l1=0 l2=2 -> L=2
        const EVec sx5_0 = vmul(s5, x0);
        EVec u5_0; vzero(u5_0);
        const EVec d5_11 = dms[11 * NQV];
        vfma(u5_0, a0.y, d5_11);
        { const float t = vdot(sx5_0, d5_11);
          dyl[4] = fmaf(1.0f, t, dyl[4]);
        }
        const EVec d5_12 = dms[12 * NQV];
        vfma(u5_0, a0.z, d5_12);
        { const float t = vdot(sx5_0, d5_12);
          dyl[5] = fmaf(1.0f, t, dyl[5]);
        }
        const EVec d5_13 = dms[13 * NQV];
        vfma(u5_0, a0.w, d5_13);
        { const float t = vdot(sx5_0, d5_13);
          dyl[6] = fmaf(1.0f, t, dyl[6]);
        }
        const EVec d5_14 = dms[14 * NQV];
        const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
        vfma(u5_0, a1.x, d5_14);
        { const float t = vdot(sx5_0, d5_14);
          dyl[7] = fmaf(1.0f, t, dyl[7]);
        }
        const EVec d5_15 = dms[15 * NQV];
        vfma(u5_0, a1.y, d5_15);
        { const float t = vdot(sx5_0, d5_15);
          dyl[8] = fmaf(1.0f, t, dyl[8]);
        }
        EVec ds5 = vmul(x0, u5_0);
        if (gw) gw[5 * NQV] = ds5;
        vfma(dxp[0], s5, u5_0);
        const EVec s6 = ss[6 * NQV];  // path 6: l1=1 l2=1 -> L=2
        const EVec sx6_1 = vmul(s6, x1);
        EVec u6_1; vzero(u6_1);
        const EVec sx6_2 = vmul(s6, x2);
        EVec u6_2; vzero(u6_2);
        const EVec sx6_3 = vmul(s6, x3);
        EVec u6_3; vzero(u6_3);
        const EVec d6_16 = dms[16 * NQV];
        vfma(u6_1, a1.z, d6_16);
        { const float t = vdot(sx6_1, d6_16);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        const EVec d6_17 = dms[17 * NQV];
        const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
        vfma(u6_1, a2.x, d6_17);
        { const float t = vdot(sx6_1, d6_17);
          dyl[2] = fmaf(0.707106769f, t, dyl[2]);
        }
        const EVec d6_18 = dms[18 * NQV];
        vfma(u6_1, a2.z, d6_18);
        { const float t = vdot(sx6_1, d6_18);
          dyl[1] = fmaf(-0.408248305f, t, dyl[1]);
        }
        const EVec d6_19 = dms[19 * NQV];
        const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
        vfma(u6_2, a3.y, d6_19);
        { const float t = vdot(sx6_2, d6_19);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        const EVec d6_20 = dms[20 * NQV];
        vfma(u6_1, a3.w, d6_20);
        { const float t = vdot(sx6_1, d6_20);
          dyl[1] = fmaf(-0.707106769f, t, dyl[1]);
        }
        vfma(u6_3, a1.w, d6_16);
        { const float t = vdot(sx6_3, d6_16);
          dyl[1] = fmaf(0.707106769f, t, dyl[1]);
        }
        vfma(u6_2, a2.y, d6_17);
        { const float t = vdot(sx6_2, d6_17);
          dyl[1] = fmaf(0.707106769f, t, dyl[1]);
        }
        vfma(u6_2, a2.w, d6_18);
        { const float t = vdot(sx6_2, d6_18);
          dyl[2] = fmaf(0.816496611f, t, dyl[2]);
        }
        vfma(u6_3, a3.z, d6_19);
        { const float t = vdot(sx6_3, d6_19);
          dyl[2] = fmaf(0.707106769f, t, dyl[2]);
        }
        const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
        vfma(u6_3, a4.x, d6_20);
        { const float t = vdot(sx6_3, d6_20);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        vfma(u6_3, a3.x, d6_18);
        { const float t = vdot(sx6_3, d6_18);
          dyl[3] = fmaf(-0.408248305f, t, dyl[3]);
        }
        EVec ds6 = vmul(x1, u6_1);
        vfma(ds6, x2, u6_2);
        vfma(ds6, x3, u6_3);
        if (gw) gw[6 * NQV] = ds6;
        vfma(dxp[1], s6, u6_1);
        vfma(dxp[2], s6, u6_2);
        vfma(dxp[3], s6, u6_3);
        const EVec s7 = ss[7 * NQV];  // path 7: l1=1 l2=3 -> L=2
        const EVec sx7_1 = vmul(s7, x1);
        EVec u7_1; vzero(u7_1);
        const EVec sx7_2 = vmul(s7, x2);
        EVec u7_2; vzero(u7_2);
        const EVec sx7_3 = vmul(s7, x3);
        EVec u7_3; vzero(u7_3);
        const EVec d7_21 = dms[21 * NQV];
        const float4 a15 = *reinterpret_cast<const float4*>(As + 60);
        vfma(u7_1, a15.x, d7_21);
        { const float t = vdot(sx7_1, d7_21);
          dyl[13] = 0.154303357f * t;
          dyl[15] = 0.597614288f * t;
        }
        const EVec d7_22 = dms[22 * NQV];
        vfma(u7_1, a15.w, d7_22);
        { const float t = vdot(sx7_1, d7_22);
          dyl[12] = 0.377964467f * t;
          dyl[14] = 0.487950027f * t;
        }
        const EVec d7_23 = dms[23 * NQV];
        const float4 a16 = *reinterpret_cast<const float4*>(As + 64);
        vfma(u7_1, a16.z, d7_23);
        { const float t = vdot(sx7_1, d7_23);
          dyl[11] = -0.534522474f * t;
        }
        const EVec d7_24 = dms[24 * NQV];
        const float4 a17 = *reinterpret_cast<const float4*>(As + 68);
        vfma(u7_1, a17.y, d7_24);
        { const float t = vdot(sx7_1, d7_24);
          dyl[10] = -0.487950027f * t;
        }
        const EVec d7_25 = dms[25 * NQV];
        const float4 a18 = *reinterpret_cast<const float4*>(As + 72);
        vfma(u7_1, a18.x, d7_25);
        { const float t = vdot(sx7_1, d7_25);
          dyl[9] = -0.597614288f * t;
          dyl[11] = fmaf(-0.154303357f, t, dyl[11]);
        }
        vfma(u7_2, a15.y, d7_21);
        { const float t = vdot(sx7_2, d7_21);
          dyl[10] = fmaf(-0.487950027f, t, dyl[10]);
        }
        vfma(u7_2, a16.x, d7_22);
        { const float t = vdot(sx7_2, d7_22);
          dyl[11] = fmaf(-0.617213428f, t, dyl[11]);
        }
        vfma(u7_2, a16.w, d7_23);
        { const float t = vdot(sx7_2, d7_23);
          dyl[12] = fmaf(-0.654653668f, t, dyl[12]);
        }
        vfma(u7_2, a17.z, d7_24);
        { const float t = vdot(sx7_2, d7_24);
          dyl[13] = fmaf(-0.617213428f, t, dyl[13]);
        }
        vfma(u7_2, a18.y, d7_25);
        { const float t = vdot(sx7_2, d7_25);
          dyl[14] = fmaf(-0.487950027f, t, dyl[14]);
        }
        vfma(u7_3, a15.z, d7_21);
        { const float t = vdot(sx7_3, d7_21);
          dyl[9] = fmaf(-0.597614288f, t, dyl[9]);
          dyl[11] = fmaf(0.154303357f, t, dyl[11]);
        }
        vfma(u7_3, a16.y, d7_22);
        { const float t = vdot(sx7_3, d7_22);
          dyl[10] = fmaf(-0.487950027f, t, dyl[10]);
        }
        vfma(u7_3, a17.x, d7_23);
        { const float t = vdot(sx7_3, d7_23);
          dyl[13] = fmaf(-0.534522474f, t, dyl[13]);
        }
        vfma(u7_3, a17.w, d7_24);
        { const float t = vdot(sx7_3, d7_24);
          dyl[12] = fmaf(0.377964467f, t, dyl[12]);
          dyl[14] = fmaf(-0.487950027f, t, dyl[14]);
        }
        vfma(u7_3, a18.z, d7_25);
        { const float t = vdot(sx7_3, d7_25);
          dyl[13] = fmaf(0.154303357f, t, dyl[13]);
          dyl[15] = fmaf(-0.597614288f, t, dyl[15]);
        }
        EVec ds7 = vmul(x1, u7_1);
        vfma(ds7, x2, u7_2);
        vfma(ds7, x3, u7_3);
        if (gw) gw[7 * NQV] = ds7;
        vfma(dxp[1], s7, u7_1);
        vfma(dxp[2], s7, u7_2);
        vfma(dxp[3], s7, u7_3);
        const EVec s8 = ss[8 * NQV];  // path 8: l1=0 l2=3 -> L=3
        const EVec sx8_0 = vmul(s8, x0);
        EVec u8_0; vzero(u8_0);
        const EVec d8_26 = dms[26 * NQV];
        vfma(u8_0, a18.w, d8_26);
        { const float t = vdot(sx8_0, d8_26);
          dyl[9] = fmaf(1.0f, t, dyl[9]);
        }
        const EVec d8_27 = dms[27 * NQV];
        const float4 a19 = *reinterpret_cast<const float4*>(As + 76);
        vfma(u8_0, a19.x, d8_27);
        { const float t = vdot(sx8_0, d8_27);
          dyl[10] = fmaf(1.0f, t, dyl[10]);
        }
        const EVec d8_28 = dms[28 * NQV];
        vfma(u8_0, a19.y, d8_28);
        { const float t = vdot(sx8_0, d8_28);
          dyl[11] = fmaf(1.0f, t, dyl[11]);
        }
        const EVec d8_29 = dms[29 * NQV];
        vfma(u8_0, a19.z, d8_29);
        { const float t = vdot(sx8_0, d8_29);
          dyl[12] = fmaf(1.0f, t, dyl[12]);
        }
        const EVec d8_30 = dms[30 * NQV];
        vfma(u8_0, a19.w, d8_30);
        { const float t = vdot(sx8_0, d8_30);
          dyl[13] = fmaf(1.0f, t, dyl[13]);
        }
        const EVec d8_31 = dms[31 * NQV];
        const float4 a20 = *reinterpret_cast<const float4*>(As + 80);
        vfma(u8_0, a20.x, d8_31);
        { const float t = vdot(sx8_0, d8_31);
          dyl[14] = fmaf(1.0f, t, dyl[14]);
        }
        const EVec d8_32 = dms[32 * NQV];
        vfma(u8_0, a20.y, d8_32);
        { const float t = vdot(sx8_0, d8_32);
          dyl[15] = fmaf(1.0f, t, dyl[15]);
        }
        EVec ds8 = vmul(x0, u8_0);
        if (gw) gw[8 * NQV] = ds8;
        vfma(dxp[0], s8, u8_0);
        const EVec s9 = ss[9 * NQV];  // path 9: l1=1 l2=2 -> L=3
        const EVec sx9_1 = vmul(s9, x1);
        EVec u9_1; vzero(u9_1);
        const EVec sx9_2 = vmul(s9, x2);
        EVec u9_2; vzero(u9_2);
        const EVec sx9_3 = vmul(s9, x3);
        EVec u9_3; vzero(u9_3);
        const EVec d9_33 = dms[33 * NQV];
        vfma(u9_1, a9.w, d9_33);
        { const float t = vdot(sx9_1, d9_33);
          dyl[8] = fmaf(0.707106769f, t, dyl[8]);
        }
        const EVec d9_34 = dms[34 * NQV];
        const float4 a10 = *reinterpret_cast<const float4*>(As + 40);
        vfma(u9_1, a10.y, d9_34);
        { const float t = vdot(sx9_1, d9_34);
          dyl[7] = fmaf(0.577350259f, t, dyl[7]);
        }
        const EVec d9_35 = dms[35 * NQV];
        const float4 a11 = *reinterpret_cast<const float4*>(As + 44);
        vfma(u9_1, a11.x, d9_35);
        { const float t = vdot(sx9_1, d9_35);
          dyl[6] = fmaf(0.632455528f, t, dyl[6]);
          dyl[8] = fmaf(0.182574183f, t, dyl[8]);
        }
        const EVec d9_36 = dms[36 * NQV];
        vfma(u9_1, a11.w, d9_36);
        { const float t = vdot(sx9_1, d9_36);
          dyl[5] = fmaf(-0.44721359f, t, dyl[5]);
        }
        const EVec d9_37 = dms[37 * NQV];
        const float4 a12 = *reinterpret_cast<const float4*>(As + 48);
        vfma(u9_1, a12.z, d9_37);
        { const float t = vdot(sx9_1, d9_37);
          dyl[4] = fmaf(-0.182574183f, t, dyl[4]);
        }
        const EVec d9_38 = dms[38 * NQV];
        const float4 a13 = *reinterpret_cast<const float4*>(As + 52);
        vfma(u9_1, a13.y, d9_38);
        { const float t = vdot(sx9_1, d9_38);
          dyl[5] = fmaf(-0.577350259f, t, dyl[5]);
        }
        const EVec d9_39 = dms[39 * NQV];
        const float4 a14 = *reinterpret_cast<const float4*>(As + 56);
        vfma(u9_1, a14.x, d9_39);
        { const float t = vdot(sx9_1, d9_39);
          dyl[4] = fmaf(-0.707106769f, t, dyl[4]);
        }
        vfma(u9_3, a10.x, d9_33);
        { const float t = vdot(sx9_3, d9_33);
          dyl[4] = fmaf(0.707106769f, t, dyl[4]);
        }
        vfma(u9_2, a10.z, d9_34);
        { const float t = vdot(sx9_2, d9_34);
          dyl[4] = fmaf(0.577350259f, t, dyl[4]);
        }
        vfma(u9_2, a11.y, d9_35);
        { const float t = vdot(sx9_2, d9_35);
          dyl[5] = fmaf(0.730296731f, t, dyl[5]);
        }
        vfma(u9_2, a12.x, d9_36);
        { const float t = vdot(sx9_2, d9_36);
          dyl[6] = fmaf(0.774596691f, t, dyl[6]);
        }
        vfma(u9_2, a12.w, d9_37);
        { const float t = vdot(sx9_2, d9_37);
          dyl[7] = fmaf(0.730296731f, t, dyl[7]);
        }
        vfma(u9_2, a13.z, d9_38);
        { const float t = vdot(sx9_2, d9_38);
          dyl[8] = fmaf(0.577350259f, t, dyl[8]);
        }
        vfma(u9_3, a14.y, d9_39);
        { const float t = vdot(sx9_3, d9_39);
          dyl[8] = fmaf(0.707106769f, t, dyl[8]);
        }
        vfma(u9_3, a10.w, d9_34);
        { const float t = vdot(sx9_3, d9_34);
          dyl[5] = fmaf(0.577350259f, t, dyl[5]);
        }
        vfma(u9_3, a11.z, d9_35);
        { const float t = vdot(sx9_3, d9_35);
          dyl[4] = fmaf(-0.182574183f, t, dyl[4]);
        }
        vfma(u9_3, a12.y, d9_36);
        { const float t = vdot(sx9_3, d9_36);
          dyl[7] = fmaf(-0.44721359f, t, dyl[7]);
        }
        vfma(u9_3, a13.x, d9_37);
        { const float t = vdot(sx9_3, d9_37);
          dyl[6] = fmaf(0.632455528f, t, dyl[6]);
          dyl[8] = fmaf(-0.182574183f, t, dyl[8]);
        }
        vfma(u9_3, a13.w, d9_38);
        { const float t = vdot(sx9_3, d9_38);
          dyl[7] = fmaf(0.577350259f, t, dyl[7]);
        }
        EVec ds9 = vmul(x1, u9_1);
        vfma(ds9, x2, u9_2);
        vfma(ds9, x3, u9_3);
        if (gw) gw[9 * NQV] = ds9;
        vfma(dxp[1], s9, u9_1);
        vfma(dxp[2], s9, u9_2);
        vfma(dxp[3], s9, u9_3);
    }
    __device__ static __forceinline__ void bwd2_edge_all(const DVec* __restrict__ dms, const DVec* __restrict__ xs, const DVec* __restrict__ uxs, const DVec* __restrict__ ss, const DVec* __restrict__ uss, const float* __restrict__ As, const float* __restrict__ Bs, DVec (&dxp)[DIN], float (&dyl)[16], DVec* __restrict__ gw) {
        constexpr int NQV = NQ / DV;
        const DVec x0 = xs[0 * NQV];
        const DVec ux0 = uxs[0 * NQV];
        const DVec x1 = xs[1 * NQV];
        const DVec ux1 = uxs[1 * NQV];
        const DVec x2 = xs[2 * NQV];
        const DVec ux2 = uxs[2 * NQV];
        const DVec x3 = xs[3 * NQV];
        const DVec ux3 = uxs[3 * NQV];
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
        const DVec s1 = ss[1 * NQV];  // path 1: l1=1 l2=1 -> L=0
        const DVec us1 = uss[1 * NQV];
        DVec sxu1_1 = pmul(s1, ux1); pfma(sxu1_1, us1, x1);
        DVec v1_1; vzero(v1_1);
        DVec w1_1; vzero(w1_1);
        DVec sxu1_2 = pmul(s1, ux2); pfma(sxu1_2, us1, x2);
        DVec v1_2; vzero(v1_2);
        DVec w1_2; vzero(w1_2);
        DVec sxu1_3 = pmul(s1, ux3); pfma(sxu1_3, us1, x3);
        DVec v1_3; vzero(v1_3);
        DVec w1_3; vzero(w1_3);
        const DVec d1_1 = dms[1 * NQV];
        const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
        const float4 b5 = *reinterpret_cast<const float4*>(Bs + 20);
        pfma(v1_1, a5.x, d1_1);
        pfma(w1_1, b5.x, d1_1);
        { const float t = vdot(sxu1_1, d1_1);
          dyl[1] = 0.577350259f * t;
        }
        pfma(v1_2, a5.y, d1_1);
        pfma(w1_2, b5.y, d1_1);
        { const float t = vdot(sxu1_2, d1_1);
          dyl[2] = 0.577350259f * t;
        }
        pfma(v1_3, a5.z, d1_1);
        pfma(w1_3, b5.z, d1_1);
        { const float t = vdot(sxu1_3, d1_1);
          dyl[3] = 0.577350259f * t;
        }
        DVec ds1 = pmul(ux1, v1_1); pfma(ds1, x1, w1_1);
        pfma(ds1, ux2, v1_2); pfma(ds1, x2, w1_2);
        pfma(ds1, ux3, v1_3); pfma(ds1, x3, w1_3);
        if (gw) gw[1 * NQV] = ds1;
        dxp[1] = pmul(us1, v1_1); pfma(dxp[1], s1, w1_1);
        dxp[2] = pmul(us1, v1_2); pfma(dxp[2], s1, w1_2);
        dxp[3] = pmul(us1, v1_3); pfma(dxp[3], s1, w1_3);
        const DVec s2 = ss[2 * NQV];  // path 2: l1=0 l2=1 -> L=1
        const DVec us2 = uss[2 * NQV];
        DVec sxu2_0 = pmul(s2, ux0); pfma(sxu2_0, us2, x0);
        DVec v2_0; vzero(v2_0);
        DVec w2_0; vzero(w2_0);
        const DVec d2_2 = dms[2 * NQV];
        const float4 a9 = *reinterpret_cast<const float4*>(As + 36);
        const float4 b9 = *reinterpret_cast<const float4*>(Bs + 36);
        pfma(v2_0, a9.x, d2_2);
        pfma(w2_0, b9.x, d2_2);
        { const float t = vdot(sxu2_0, d2_2);
          dyl[1] = fmaf(1.0f, t, dyl[1]);
        }
        const DVec d2_3 = dms[3 * NQV];
        pfma(v2_0, a9.y, d2_3);
        pfma(w2_0, b9.y, d2_3);
        { const float t = vdot(sxu2_0, d2_3);
          dyl[2] = fmaf(1.0f, t, dyl[2]);
        }
        const DVec d2_4 = dms[4 * NQV];
        pfma(v2_0, a9.z, d2_4);
        pfma(w2_0, b9.z, d2_4);
        { const float t = vdot(sxu2_0, d2_4);
          dyl[3] = fmaf(1.0f, t, dyl[3]);
        }
        DVec ds2 = pmul(ux0, v2_0); pfma(ds2, x0, w2_0);
        if (gw) gw[2 * NQV] = ds2;
        pfma(dxp[0], us2, v2_0); pfma(dxp[0], s2, w2_0);
        const DVec s3 = ss[3 * NQV];  // path 3: l1=1 l2=0 -> L=1
        const DVec us3 = uss[3 * NQV];
        DVec sxu3_1 = pmul(s3, ux1); pfma(sxu3_1, us3, x1);
        DVec v3_1; vzero(v3_1);
        DVec w3_1; vzero(w3_1);
        DVec sxu3_2 = pmul(s3, ux2); pfma(sxu3_2, us3, x2);
        DVec v3_2; vzero(v3_2);
        DVec w3_2; vzero(w3_2);
        DVec sxu3_3 = pmul(s3, ux3); pfma(sxu3_3, us3, x3);
        DVec v3_3; vzero(v3_3);
        DVec w3_3; vzero(w3_3);
        const DVec d3_5 = dms[5 * NQV];
        pfma(v3_1, a5.w, d3_5);
        pfma(w3_1, b5.w, d3_5);
        { const float t = vdot(sxu3_1, d3_5);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        const DVec d3_6 = dms[6 * NQV];
        const float4 a6 = *reinterpret_cast<const float4*>(As + 24);
        const float4 b6 = *reinterpret_cast<const float4*>(Bs + 24);
        pfma(v3_2, a6.x, d3_6);
        pfma(w3_2, b6.x, d3_6);
        { const float t = vdot(sxu3_2, d3_6);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        const DVec d3_7 = dms[7 * NQV];
        pfma(v3_3, a6.y, d3_7);
        pfma(w3_3, b6.y, d3_7);
        { const float t = vdot(sxu3_3, d3_7);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        DVec ds3 = pmul(ux1, v3_1); pfma(ds3, x1, w3_1);
        pfma(ds3, ux2, v3_2); pfma(ds3, x2, w3_2);
        pfma(ds3, ux3, v3_3); pfma(ds3, x3, w3_3);
        if (gw) gw[3 * NQV] = ds3;
        pfma(dxp[1], us3, v3_1); pfma(dxp[1], s3, w3_1);
        pfma(dxp[2], us3, v3_2); pfma(dxp[2], s3, w3_2);
        pfma(dxp[3], us3, v3_3); pfma(dxp[3], s3, w3_3);
        const DVec s4 = ss[4 * NQV];  // path 4: l1=1 l2=2 -> L=1
        const DVec us4 = uss[4 * NQV];
        DVec sxu4_1 = pmul(s4, ux1); pfma(sxu4_1, us4, x1);
        DVec v4_1; vzero(v4_1);
        DVec w4_1; vzero(w4_1);
        DVec sxu4_2 = pmul(s4, ux2); pfma(sxu4_2, us4, x2);
        DVec v4_2; vzero(v4_2);
        DVec w4_2; vzero(w4_2);
        DVec sxu4_3 = pmul(s4, ux3); pfma(sxu4_3, us4, x3);
        DVec v4_3; vzero(v4_3);
        DVec w4_3; vzero(w4_3);
        const DVec d4_8 = dms[8 * NQV];
        pfma(v4_1, a6.z, d4_8);
        pfma(w4_1, b6.z, d4_8);
        { const float t = vdot(sxu4_1, d4_8);
          dyl[6] = 0.316227764f * t;
          dyl[8] = 0.547722578f * t;
        }
        const DVec d4_9 = dms[9 * NQV];
        const float4 a7 = *reinterpret_cast<const float4*>(As + 28);
        const float4 b7 = *reinterpret_cast<const float4*>(Bs + 28);
        pfma(v4_1, a7.y, d4_9);
        pfma(w4_1, b7.y, d4_9);
        { const float t = vdot(sxu4_1, d4_9);
          dyl[5] = -0.547722578f * t;
        }
        const DVec d4_10 = dms[10 * NQV];
        const float4 a8 = *reinterpret_cast<const float4*>(As + 32);
        const float4 b8 = *reinterpret_cast<const float4*>(Bs + 32);
        pfma(v4_1, a8.x, d4_10);
        pfma(w4_1, b8.x, d4_10);
        { const float t = vdot(sxu4_1, d4_10);
          dyl[4] = -0.547722578f * t;
        }
        pfma(v4_2, a6.w, d4_8);
        pfma(w4_2, b6.w, d4_8);
        { const float t = vdot(sxu4_2, d4_8);
          dyl[5] = fmaf(-0.547722578f, t, dyl[5]);
        }
        pfma(v4_2, a7.z, d4_9);
        pfma(w4_2, b7.z, d4_9);
        { const float t = vdot(sxu4_2, d4_9);
          dyl[6] = fmaf(-0.632455528f, t, dyl[6]);
        }
        pfma(v4_2, a8.y, d4_10);
        pfma(w4_2, b8.y, d4_10);
        { const float t = vdot(sxu4_2, d4_10);
          dyl[7] = -0.547722578f * t;
        }
        pfma(v4_3, a7.x, d4_8);
        pfma(w4_3, b7.x, d4_8);
        { const float t = vdot(sxu4_3, d4_8);
          dyl[4] = fmaf(-0.547722578f, t, dyl[4]);
        }
        pfma(v4_3, a7.w, d4_9);
        pfma(w4_3, b7.w, d4_9);
        { const float t = vdot(sxu4_3, d4_9);
          dyl[7] = fmaf(-0.547722578f, t, dyl[7]);
        }
        pfma(v4_3, a8.z, d4_10);
        pfma(w4_3, b8.z, d4_10);
        { const float t = vdot(sxu4_3, d4_10);
          dyl[6] = fmaf(0.316227764f, t, dyl[6]);
          dyl[8] = fmaf(-0.547722578f, t, dyl[8]);
        }
        DVec ds4 = pmul(ux1, v4_1); pfma(ds4, x1, w4_1);
        pfma(ds4, ux2, v4_2); pfma(ds4, x2, w4_2);
        pfma(ds4, ux3, v4_3); pfma(ds4, x3, w4_3);
        if (gw) gw[4 * NQV] = ds4;
        pfma(dxp[1], us4, v4_1); pfma(dxp[1], s4, w4_1);
        pfma(dxp[2], us4, v4_2); pfma(dxp[2], s4, w4_2);
        pfma(dxp[3], us4, v4_3); pfma(dxp[3], s4, w4_3);
        const DVec s5 = ss[5 * NQV];  // path 5: l1=0 l2=2 -> L=2
        const DVec us5 = uss[5 * NQV];
        DVec sxu5_0 = pmul(s5, ux0); pfma(sxu5_0, us5, x0);
        DVec v5_0; vzero(v5_0);
        DVec w5_0; vzero(w5_0);
        const DVec d5_11 = dms[11 * NQV];
        pfma(v5_0, a0.y, d5_11);
        pfma(w5_0, b0.y, d5_11);
        { const float t = vdot(sxu5_0, d5_11);
          dyl[4] = fmaf(1.0f, t, dyl[4]);
        }
        const DVec d5_12 = dms[12 * NQV];
        pfma(v5_0, a0.z, d5_12);
        pfma(w5_0, b0.z, d5_12);
        { const float t = vdot(sxu5_0, d5_12);
          dyl[5] = fmaf(1.0f, t, dyl[5]);
        }
        const DVec d5_13 = dms[13 * NQV];
        pfma(v5_0, a0.w, d5_13);
        pfma(w5_0, b0.w, d5_13);
        { const float t = vdot(sxu5_0, d5_13);
          dyl[6] = fmaf(1.0f, t, dyl[6]);
        }
        const DVec d5_14 = dms[14 * NQV];
        const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
        const float4 b1 = *reinterpret_cast<const float4*>(Bs + 4);
        pfma(v5_0, a1.x, d5_14);
        pfma(w5_0, b1.x, d5_14);
        { const float t = vdot(sxu5_0, d5_14);
          dyl[7] = fmaf(1.0f, t, dyl[7]);
        }
        const DVec d5_15 = dms[15 * NQV];
        pfma(v5_0, a1.y, d5_15);
        pfma(w5_0, b1.y, d5_15);
        { const float t = vdot(sxu5_0, d5_15);
          dyl[8] = fmaf(1.0f, t, dyl[8]);
        }
        DVec ds5 = pmul(ux0, v5_0); pfma(ds5, x0, w5_0);
        if (gw) gw[5 * NQV] = ds5;
        pfma(dxp[0], us5, v5_0); pfma(dxp[0], s5, w5_0);
        const DVec s6 = ss[6 * NQV];  // path 6: l1=1 l2=1 -> L=2
        const DVec us6 = uss[6 * NQV];
        DVec sxu6_1 = pmul(s6, ux1); pfma(sxu6_1, us6, x1);
        DVec v6_1; vzero(v6_1);
        DVec w6_1; vzero(w6_1);
        DVec sxu6_2 = pmul(s6, ux2); pfma(sxu6_2, us6, x2);
        DVec v6_2; vzero(v6_2);
        DVec w6_2; vzero(w6_2);
        DVec sxu6_3 = pmul(s6, ux3); pfma(sxu6_3, us6, x3);
        DVec v6_3; vzero(v6_3);
        DVec w6_3; vzero(w6_3);
        const DVec d6_16 = dms[16 * NQV];
        pfma(v6_1, a1.z, d6_16);
        pfma(w6_1, b1.z, d6_16);
        { const float t = vdot(sxu6_1, d6_16);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        const DVec d6_17 = dms[17 * NQV];
        const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
        const float4 b2 = *reinterpret_cast<const float4*>(Bs + 8);
        pfma(v6_1, a2.x, d6_17);
        pfma(w6_1, b2.x, d6_17);
        { const float t = vdot(sxu6_1, d6_17);
          dyl[2] = fmaf(0.707106769f, t, dyl[2]);
        }
        const DVec d6_18 = dms[18 * NQV];
        pfma(v6_1, a2.z, d6_18);
        pfma(w6_1, b2.z, d6_18);
        { const float t = vdot(sxu6_1, d6_18);
          dyl[1] = fmaf(-0.408248305f, t, dyl[1]);
        }
        const DVec d6_19 = dms[19 * NQV];
        const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
        const float4 b3 = *reinterpret_cast<const float4*>(Bs + 12);
        pfma(v6_2, a3.y, d6_19);
        pfma(w6_2, b3.y, d6_19);
        { const float t = vdot(sxu6_2, d6_19);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        const DVec d6_20 = dms[20 * NQV];
        pfma(v6_1, a3.w, d6_20);
        pfma(w6_1, b3.w, d6_20);
        { const float t = vdot(sxu6_1, d6_20);
          dyl[1] = fmaf(-0.707106769f, t, dyl[1]);
        }
        pfma(v6_3, a1.w, d6_16);
        pfma(w6_3, b1.w, d6_16);
        { const float t = vdot(sxu6_3, d6_16);
          dyl[1] = fmaf(0.707106769f, t, dyl[1]);
        }
        pfma(v6_2, a2.y, d6_17);
        pfma(w6_2, b2.y, d6_17);
        { const float t = vdot(sxu6_2, d6_17);
          dyl[1] = fmaf(0.707106769f, t, dyl[1]);
        }
        pfma(v6_2, a2.w, d6_18);
        pfma(w6_2, b2.w, d6_18);
        { const float t = vdot(sxu6_2, d6_18);
          dyl[2] = fmaf(0.816496611f, t, dyl[2]);
        }
        pfma(v6_3, a3.z, d6_19);
        pfma(w6_3, b3.z, d6_19);
        { const float t = vdot(sxu6_3, d6_19);
          dyl[2] = fmaf(0.707106769f, t, dyl[2]);
        }
        const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
        const float4 b4 = *reinterpret_cast<const float4*>(Bs + 16);
        pfma(v6_3, a4.x, d6_20);
        pfma(w6_3, b4.x, d6_20);
        { const float t = vdot(sxu6_3, d6_20);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        pfma(v6_3, a3.x, d6_18);
        pfma(w6_3, b3.x, d6_18);
        { const float t = vdot(sxu6_3, d6_18);
          dyl[3] = fmaf(-0.408248305f, t, dyl[3]);
        }
        DVec ds6 = pmul(ux1, v6_1); pfma(ds6, x1, w6_1);
        pfma(ds6, ux2, v6_2); pfma(ds6, x2, w6_2);
        pfma(ds6, ux3, v6_3); pfma(ds6, x3, w6_3);
        if (gw) gw[6 * NQV] = ds6;
        pfma(dxp[1], us6, v6_1); pfma(dxp[1], s6, w6_1);
        pfma(dxp[2], us6, v6_2); pfma(dxp[2], s6, w6_2);
        pfma(dxp[3], us6, v6_3); pfma(dxp[3], s6, w6_3);
        const DVec s7 = ss[7 * NQV];  // path 7: l1=1 l2=3 -> L=2
        const DVec us7 = uss[7 * NQV];
        DVec sxu7_1 = pmul(s7, ux1); pfma(sxu7_1, us7, x1);
        DVec v7_1; vzero(v7_1);
        DVec w7_1; vzero(w7_1);
        DVec sxu7_2 = pmul(s7, ux2); pfma(sxu7_2, us7, x2);
        DVec v7_2; vzero(v7_2);
        DVec w7_2; vzero(w7_2);
        DVec sxu7_3 = pmul(s7, ux3); pfma(sxu7_3, us7, x3);
        DVec v7_3; vzero(v7_3);
        DVec w7_3; vzero(w7_3);
        const DVec d7_21 = dms[21 * NQV];
        const float4 a15 = *reinterpret_cast<const float4*>(As + 60);
        const float4 b15 = *reinterpret_cast<const float4*>(Bs + 60);
        pfma(v7_1, a15.x, d7_21);
        pfma(w7_1, b15.x, d7_21);
        { const float t = vdot(sxu7_1, d7_21);
          dyl[13] = 0.154303357f * t;
          dyl[15] = 0.597614288f * t;
        }
        const DVec d7_22 = dms[22 * NQV];
        pfma(v7_1, a15.w, d7_22);
        pfma(w7_1, b15.w, d7_22);
        { const float t = vdot(sxu7_1, d7_22);
          dyl[12] = 0.377964467f * t;
          dyl[14] = 0.487950027f * t;
        }
        const DVec d7_23 = dms[23 * NQV];
        const float4 a16 = *reinterpret_cast<const float4*>(As + 64);
        const float4 b16 = *reinterpret_cast<const float4*>(Bs + 64);
        pfma(v7_1, a16.z, d7_23);
        pfma(w7_1, b16.z, d7_23);
        { const float t = vdot(sxu7_1, d7_23);
          dyl[11] = -0.534522474f * t;
        }
        const DVec d7_24 = dms[24 * NQV];
        const float4 a17 = *reinterpret_cast<const float4*>(As + 68);
        const float4 b17 = *reinterpret_cast<const float4*>(Bs + 68);
        pfma(v7_1, a17.y, d7_24);
        pfma(w7_1, b17.y, d7_24);
        { const float t = vdot(sxu7_1, d7_24);
          dyl[10] = -0.487950027f * t;
        }
        const DVec d7_25 = dms[25 * NQV];
        const float4 a18 = *reinterpret_cast<const float4*>(As + 72);
        const float4 b18 = *reinterpret_cast<const float4*>(Bs + 72);
        pfma(v7_1, a18.x, d7_25);
        pfma(w7_1, b18.x, d7_25);
        { const float t = vdot(sxu7_1, d7_25);
          dyl[9] = -0.597614288f * t;
          dyl[11] = fmaf(-0.154303357f, t, dyl[11]);
        }
        pfma(v7_2, a15.y, d7_21);
        pfma(w7_2, b15.y, d7_21);
        { const float t = vdot(sxu7_2, d7_21);
          dyl[10] = fmaf(-0.487950027f, t, dyl[10]);
        }
        pfma(v7_2, a16.x, d7_22);
        pfma(w7_2, b16.x, d7_22);
        { const float t = vdot(sxu7_2, d7_22);
          dyl[11] = fmaf(-0.617213428f, t, dyl[11]);
        }
        pfma(v7_2, a16.w, d7_23);
        pfma(w7_2, b16.w, d7_23);
        { const float t = vdot(sxu7_2, d7_23);
          dyl[12] = fmaf(-0.654653668f, t, dyl[12]);
        }
        pfma(v7_2, a17.z, d7_24);
        pfma(w7_2, b17.z, d7_24);
        { const float t = vdot(sxu7_2, d7_24);
          dyl[13] = fmaf(-0.617213428f, t, dyl[13]);
        }
        pfma(v7_2, a18.y, d7_25);
        pfma(w7_2, b18.y, d7_25);
        { const float t = vdot(sxu7_2, d7_25);
          dyl[14] = fmaf(-0.487950027f, t, dyl[14]);
        }
        pfma(v7_3, a15.z, d7_21);
        pfma(w7_3, b15.z, d7_21);
        { const float t = vdot(sxu7_3, d7_21);
          dyl[9] = fmaf(-0.597614288f, t, dyl[9]);
          dyl[11] = fmaf(0.154303357f, t, dyl[11]);
        }
        pfma(v7_3, a16.y, d7_22);
        pfma(w7_3, b16.y, d7_22);
        { const float t = vdot(sxu7_3, d7_22);
          dyl[10] = fmaf(-0.487950027f, t, dyl[10]);
        }
        pfma(v7_3, a17.x, d7_23);
        pfma(w7_3, b17.x, d7_23);
        { const float t = vdot(sxu7_3, d7_23);
          dyl[13] = fmaf(-0.534522474f, t, dyl[13]);
        }
        pfma(v7_3, a17.w, d7_24);
        pfma(w7_3, b17.w, d7_24);
        { const float t = vdot(sxu7_3, d7_24);
          dyl[12] = fmaf(0.377964467f, t, dyl[12]);
          dyl[14] = fmaf(-0.487950027f, t, dyl[14]);
        }
        pfma(v7_3, a18.z, d7_25);
        pfma(w7_3, b18.z, d7_25);
        { const float t = vdot(sxu7_3, d7_25);
          dyl[13] = fmaf(0.154303357f, t, dyl[13]);
          dyl[15] = fmaf(-0.597614288f, t, dyl[15]);
        }
        DVec ds7 = pmul(ux1, v7_1); pfma(ds7, x1, w7_1);
        pfma(ds7, ux2, v7_2); pfma(ds7, x2, w7_2);
        pfma(ds7, ux3, v7_3); pfma(ds7, x3, w7_3);
        if (gw) gw[7 * NQV] = ds7;
        pfma(dxp[1], us7, v7_1); pfma(dxp[1], s7, w7_1);
        pfma(dxp[2], us7, v7_2); pfma(dxp[2], s7, w7_2);
        pfma(dxp[3], us7, v7_3); pfma(dxp[3], s7, w7_3);
        const DVec s8 = ss[8 * NQV];  // path 8: l1=0 l2=3 -> L=3
        const DVec us8 = uss[8 * NQV];
        DVec sxu8_0 = pmul(s8, ux0); pfma(sxu8_0, us8, x0);
        DVec v8_0; vzero(v8_0);
        DVec w8_0; vzero(w8_0);
        const DVec d8_26 = dms[26 * NQV];
        pfma(v8_0, a18.w, d8_26);
        pfma(w8_0, b18.w, d8_26);
        { const float t = vdot(sxu8_0, d8_26);
          dyl[9] = fmaf(1.0f, t, dyl[9]);
        }
        const DVec d8_27 = dms[27 * NQV];
        const float4 a19 = *reinterpret_cast<const float4*>(As + 76);
        const float4 b19 = *reinterpret_cast<const float4*>(Bs + 76);
        pfma(v8_0, a19.x, d8_27);
        pfma(w8_0, b19.x, d8_27);
        { const float t = vdot(sxu8_0, d8_27);
          dyl[10] = fmaf(1.0f, t, dyl[10]);
        }
        const DVec d8_28 = dms[28 * NQV];
        pfma(v8_0, a19.y, d8_28);
        pfma(w8_0, b19.y, d8_28);
        { const float t = vdot(sxu8_0, d8_28);
          dyl[11] = fmaf(1.0f, t, dyl[11]);
        }
        const DVec d8_29 = dms[29 * NQV];
        pfma(v8_0, a19.z, d8_29);
        pfma(w8_0, b19.z, d8_29);
        { const float t = vdot(sxu8_0, d8_29);
          dyl[12] = fmaf(1.0f, t, dyl[12]);
        }
        const DVec d8_30 = dms[30 * NQV];
        pfma(v8_0, a19.w, d8_30);
        pfma(w8_0, b19.w, d8_30);
        { const float t = vdot(sxu8_0, d8_30);
          dyl[13] = fmaf(1.0f, t, dyl[13]);
        }
        const DVec d8_31 = dms[31 * NQV];
        const float4 a20 = *reinterpret_cast<const float4*>(As + 80);
        const float4 b20 = *reinterpret_cast<const float4*>(Bs + 80);
        pfma(v8_0, a20.x, d8_31);
        pfma(w8_0, b20.x, d8_31);
        { const float t = vdot(sxu8_0, d8_31);
          dyl[14] = fmaf(1.0f, t, dyl[14]);
        }
        const DVec d8_32 = dms[32 * NQV];
        pfma(v8_0, a20.y, d8_32);
        pfma(w8_0, b20.y, d8_32);
        { const float t = vdot(sxu8_0, d8_32);
          dyl[15] = fmaf(1.0f, t, dyl[15]);
        }
        DVec ds8 = pmul(ux0, v8_0); pfma(ds8, x0, w8_0);
        if (gw) gw[8 * NQV] = ds8;
        pfma(dxp[0], us8, v8_0); pfma(dxp[0], s8, w8_0);
        const DVec s9 = ss[9 * NQV];  // path 9: l1=1 l2=2 -> L=3
        const DVec us9 = uss[9 * NQV];
        DVec sxu9_1 = pmul(s9, ux1); pfma(sxu9_1, us9, x1);
        DVec v9_1; vzero(v9_1);
        DVec w9_1; vzero(w9_1);
        DVec sxu9_2 = pmul(s9, ux2); pfma(sxu9_2, us9, x2);
        DVec v9_2; vzero(v9_2);
        DVec w9_2; vzero(w9_2);
        DVec sxu9_3 = pmul(s9, ux3); pfma(sxu9_3, us9, x3);
        DVec v9_3; vzero(v9_3);
        DVec w9_3; vzero(w9_3);
        const DVec d9_33 = dms[33 * NQV];
        pfma(v9_1, a9.w, d9_33);
        pfma(w9_1, b9.w, d9_33);
        { const float t = vdot(sxu9_1, d9_33);
          dyl[8] = fmaf(0.707106769f, t, dyl[8]);
        }
        const DVec d9_34 = dms[34 * NQV];
        const float4 a10 = *reinterpret_cast<const float4*>(As + 40);
        const float4 b10 = *reinterpret_cast<const float4*>(Bs + 40);
        pfma(v9_1, a10.y, d9_34);
        pfma(w9_1, b10.y, d9_34);
        { const float t = vdot(sxu9_1, d9_34);
          dyl[7] = fmaf(0.577350259f, t, dyl[7]);
        }
        const DVec d9_35 = dms[35 * NQV];
        const float4 a11 = *reinterpret_cast<const float4*>(As + 44);
        const float4 b11 = *reinterpret_cast<const float4*>(Bs + 44);
        pfma(v9_1, a11.x, d9_35);
        pfma(w9_1, b11.x, d9_35);
        { const float t = vdot(sxu9_1, d9_35);
          dyl[6] = fmaf(0.632455528f, t, dyl[6]);
          dyl[8] = fmaf(0.182574183f, t, dyl[8]);
        }
        const DVec d9_36 = dms[36 * NQV];
        pfma(v9_1, a11.w, d9_36);
        pfma(w9_1, b11.w, d9_36);
        { const float t = vdot(sxu9_1, d9_36);
          dyl[5] = fmaf(-0.44721359f, t, dyl[5]);
        }
        const DVec d9_37 = dms[37 * NQV];
        const float4 a12 = *reinterpret_cast<const float4*>(As + 48);
        const float4 b12 = *reinterpret_cast<const float4*>(Bs + 48);
        pfma(v9_1, a12.z, d9_37);
        pfma(w9_1, b12.z, d9_37);
        { const float t = vdot(sxu9_1, d9_37);
          dyl[4] = fmaf(-0.182574183f, t, dyl[4]);
        }
        const DVec d9_38 = dms[38 * NQV];
        const float4 a13 = *reinterpret_cast<const float4*>(As + 52);
        const float4 b13 = *reinterpret_cast<const float4*>(Bs + 52);
        pfma(v9_1, a13.y, d9_38);
        pfma(w9_1, b13.y, d9_38);
        { const float t = vdot(sxu9_1, d9_38);
          dyl[5] = fmaf(-0.577350259f, t, dyl[5]);
        }
        const DVec d9_39 = dms[39 * NQV];
        const float4 a14 = *reinterpret_cast<const float4*>(As + 56);
        const float4 b14 = *reinterpret_cast<const float4*>(Bs + 56);
        pfma(v9_1, a14.x, d9_39);
        pfma(w9_1, b14.x, d9_39);
        { const float t = vdot(sxu9_1, d9_39);
          dyl[4] = fmaf(-0.707106769f, t, dyl[4]);
        }
        pfma(v9_3, a10.x, d9_33);
        pfma(w9_3, b10.x, d9_33);
        { const float t = vdot(sxu9_3, d9_33);
          dyl[4] = fmaf(0.707106769f, t, dyl[4]);
        }
        pfma(v9_2, a10.z, d9_34);
        pfma(w9_2, b10.z, d9_34);
        { const float t = vdot(sxu9_2, d9_34);
          dyl[4] = fmaf(0.577350259f, t, dyl[4]);
        }
        pfma(v9_2, a11.y, d9_35);
        pfma(w9_2, b11.y, d9_35);
        { const float t = vdot(sxu9_2, d9_35);
          dyl[5] = fmaf(0.730296731f, t, dyl[5]);
        }
        pfma(v9_2, a12.x, d9_36);
        pfma(w9_2, b12.x, d9_36);
        { const float t = vdot(sxu9_2, d9_36);
          dyl[6] = fmaf(0.774596691f, t, dyl[6]);
        }
        pfma(v9_2, a12.w, d9_37);
        pfma(w9_2, b12.w, d9_37);
        { const float t = vdot(sxu9_2, d9_37);
          dyl[7] = fmaf(0.730296731f, t, dyl[7]);
        }
        pfma(v9_2, a13.z, d9_38);
        pfma(w9_2, b13.z, d9_38);
        { const float t = vdot(sxu9_2, d9_38);
          dyl[8] = fmaf(0.577350259f, t, dyl[8]);
        }
        pfma(v9_3, a14.y, d9_39);
        pfma(w9_3, b14.y, d9_39);
        { const float t = vdot(sxu9_3, d9_39);
          dyl[8] = fmaf(0.707106769f, t, dyl[8]);
        }
        pfma(v9_3, a10.w, d9_34);
        pfma(w9_3, b10.w, d9_34);
        { const float t = vdot(sxu9_3, d9_34);
          dyl[5] = fmaf(0.577350259f, t, dyl[5]);
        }
        pfma(v9_3, a11.z, d9_35);
        pfma(w9_3, b11.z, d9_35);
        { const float t = vdot(sxu9_3, d9_35);
          dyl[4] = fmaf(-0.182574183f, t, dyl[4]);
        }
        pfma(v9_3, a12.y, d9_36);
        pfma(w9_3, b12.y, d9_36);
        { const float t = vdot(sxu9_3, d9_36);
          dyl[7] = fmaf(-0.44721359f, t, dyl[7]);
        }
        pfma(v9_3, a13.x, d9_37);
        pfma(w9_3, b13.x, d9_37);
        { const float t = vdot(sxu9_3, d9_37);
          dyl[6] = fmaf(0.632455528f, t, dyl[6]);
          dyl[8] = fmaf(-0.182574183f, t, dyl[8]);
        }
        pfma(v9_3, a13.w, d9_38);
        pfma(w9_3, b13.w, d9_38);
        { const float t = vdot(sxu9_3, d9_38);
          dyl[7] = fmaf(0.577350259f, t, dyl[7]);
        }
        DVec ds9 = pmul(ux1, v9_1); pfma(ds9, x1, w9_1);
        pfma(ds9, ux2, v9_2); pfma(ds9, x2, w9_2);
        pfma(ds9, ux3, v9_3); pfma(ds9, x3, w9_3);
        if (gw) gw[9 * NQV] = ds9;
        pfma(dxp[1], us9, v9_1); pfma(dxp[1], s9, w9_1);
        pfma(dxp[2], us9, v9_2); pfma(dxp[2], s9, w9_2);
        pfma(dxp[3], us9, v9_3); pfma(dxp[3], s9, w9_3);
    }
};
}  // namespace
}  // namespace fast

extern const FastKernels kFast_w128_l3_natural;
const FastKernels kFast_w128_l3_natural = {
    "128|0e+1o|3|0:0:0,1:1:0,0:1:1,1:0:1,1:2:1,0:2:2,1:1:2,1:3:2,0:3:3,1:2:3",
    &fast::fwd_scratch_bytes<fast::Sig_w128_l3_natural>, &fast::bwd_scratch_bytes<fast::Sig_w128_l3_natural>, &fast::launch_fwd<fast::Sig_w128_l3_natural>, &fast::launch_bwd<fast::Sig_w128_l3_natural>, &fast::launch_tp_fwd<fast::Sig_w128_l3_natural>, &fast::launch_tp_bwd<fast::Sig_w128_l3_natural>,
    &fast::launch_dbl_edges<fast::Sig_w128_l3_natural>, &fast::launch_dbl_out<fast::Sig_w128_l3_natural>, nullptr, &fast::launch_bwd_sched<fast::Sig_w128_l3_natural>, 11};
}  // namespace e3j
