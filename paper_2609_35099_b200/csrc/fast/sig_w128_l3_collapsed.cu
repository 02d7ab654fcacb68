// GENERATED by csrc/gen_fast.py from fast/signatures.json -- do not edit.
// signature: 128|0e+1o|3|0:0:0,1:1:0,0:1:1,1:0:1,1:2:1,1:1:1,0:2:2,1:1:2,1:3:2,1:2:2,0:3:3,1:2:3,1:3:3|collapsed
// 128x0e+128x1o (x) harmonics l<=3: P=13 D=31 nnz=134 pairs=116
#include "fast_fwd.cuh"
#include "fast_bwd.cuh"
#include "fast_launch.cuh"

namespace e3j {
namespace fast {
namespace {
__device__ const PairRec kPair_w128_l3_collapsed[124] = {
    {0,1}, {1,1}, {2,1}, {3,1}, {4,1}, {5,1}, {6,2}, {8,1}, {9,1}, {10,1}, {11,1}, {12,1}, {13,1}, {14,1}, {15,1}, {16,1}, {17,1}, {18,1}, {19,2}, {21,1}, {22,1}, {23,0}, {23,0}, {23,0}, {23,1}, {24,1}, {25,1}, {26,1}, {27,1}, {28,1}, {29,1}, {30,2}, {32,1}, {33,2}, {35,1}, {36,1}, {37,1}, {38,2}, {40,1}, {41,1}, {42,1}, {43,1}, {44,1}, {45,1}, {46,1}, {47,1}, {48,1}, {49,1}, {50,1}, {51,1}, {52,1}, {53,1}, {54,2}, {56,0}, {56,0}, {56,0}, {56,1}, {57,1}, {58,1}, {59,2}, {61,1}, {62,2}, {64,1}, {65,1}, {66,1}, {67,1}, {68,1}, {69,2}, {71,1}, {72,1}, {73,2}, {75,1}, {76,1}, {77,1}, {78,1}, {79,1}, {80,1}, {81,1}, {82,1}, {83,1}, {84,1}, {85,1}, {86,1}, {87,1}, {88,2}, {90,1}, {91,1}, {92,0}, {92,1}, {93,1}, {94,1}, {95,1}, {96,1}, {97,1}, {98,1}, {99,2}, {101,1}, {102,1}, {103,1}, {104,1}, {105,1}, {106,1}, {107,1}, {108,1}, {109,1}, {110,1}, {111,2}, {113,1}, {114,2}, {116,1}, {117,1}, {118,2}, {120,1}, {121,1}, {122,2}, {124,1}, {125,1}, {126,2}, {128,1}, {129,2}, {131,1}, {132,1}, {133,1}, {134,0}};
__device__ const float kVal_w128_l3_collapsed[134] = {
    1.0f, 0.577350259f, 0.577350259f, 0.577350259f, 1.0f, 1.0f, 0.316227764f, 0.547722578f, -0.547722578f, -0.547722578f, 1.0f, 1.0f, -0.547722578f, -0.632455528f, -0.547722578f, 1.0f, 1.0f, -0.547722578f, -0.547722578f, 0.316227764f, -0.547722578f, 0.707106769f, -0.707106769f, -0.707106769f, 0.707106769f, 0.707106769f, -0.707106769f, 1.0f, 0.707106769f, 0.707106769f, 0.154303357f, 0.597614288f, -0.487950027f, -0.597614288f, 0.154303357f, 1.0f, 0.707106769f, 0.707106769f, 0.377964467f, 0.487950027f, -0.617213428f, -0.487950027f, 1.0f, -0.408248305f, 0.816496611f, -0.408248305f, -0.534522474f, -0.654653668f, -0.534522474f, 1.0f, 0.707106769f, 0.707106769f, -0.487950027f, -0.617213428f, 0.377964467f, -0.487950027f, 1.0f, -0.707106769f, 0.707106769f, -0.597614288f, -0.154303357f, -0.487950027f, 0.154303357f, -0.597614288f, 0.408248305f, 0.816496611f, -0.408248305f, -0.408248305f, 0.408248305f, -0.707106769f, -0.408248305f, -0.707106769f, 0.707106769f, 0.707106769f, -0.408248305f, -0.408248305f, 0.408248305f, 0.408248305f, -0.816496611f, 0.408248305f, 1.0f, 0.707106769f, 0.707106769f, 1.0f, 0.577350259f, 0.577350259f, 0.577350259f, 1.0f, 0.632455528f, 0.182574183f, 0.730296731f, -0.182574183f, 1.0f, -0.44721359f, 0.774596691f, -0.44721359f, 1.0f, -0.182574183f, 0.730296731f, 0.632455528f, -0.182574183f, 1.0f, -0.577350259f, 0.577350259f, 0.577350259f, 1.0f, -0.707106769f, 0.707106769f, 0.353553385f, 0.866025388f, -0.353553385f, -0.353553385f, 0.456435472f, 0.577350259f, -0.456435472f, -0.353553385f, -0.456435472f, 0.288675129f, -0.707106769f, -0.456435472f, -0.707106769f, 0.707106769f, 0.707106769f, -0.456435472f, -0.288675129f, 0.456435472f, 0.456435472f, -0.353553385f, -0.577350259f, 0.353553385f, 0.456435472f, 0.353553385f, -0.866025388f, 0.353553385f};
__device__ const unsigned char kI2_w128_l3_collapsed[134] = {
    0, 1, 2, 3, 1, 0, 6, 8, 5, 4, 2, 0, 5, 6, 7, 3, 0, 4, 7, 6, 8, 3, 2, 3, 1, 2, 1, 4, 3, 1, 13, 15, 10, 9, 11, 5, 2, 1, 12, 14, 11, 10, 6, 1, 2, 3, 11, 12, 13, 7, 3, 2, 10, 13, 12, 14, 8, 1, 3, 9, 11, 14, 13, 15, 5, 8, 7, 4, 7, 6, 8, 7, 5, 6, 8, 5, 4, 7, 4, 5, 9, 8, 4, 10, 7, 4, 5, 11, 6, 8, 5, 4, 12, 5, 6, 7, 13, 4, 7, 6, 8, 14, 5, 8, 7, 15, 4, 8, 10, 15, 14, 9, 11, 14, 13, 15, 10, 13, 12, 14, 13, 11, 12, 14, 11, 10, 13, 15, 10, 9, 11, 14, 9, 10};
__device__ const PairRec kBPair_w128_l3_collapsed[124] = {
    {0,1}, {1,1}, {2,1}, {3,1}, {4,1}, {5,1}, {6,1}, {7,1}, {8,1}, {9,1}, {10,1}, {11,1}, {12,1}, {13,1}, {14,1}, {15,1}, {16,1}, {17,1}, {18,1}, {19,1}, {20,2}, {22,1}, {23,1}, {24,2}, {26,1}, {27,1}, {28,1}, {29,1}, {30,1}, {31,0}, {31,0}, {31,0}, {31,1}, {32,1}, {33,1}, {34,1}, {35,1}, {36,1}, {37,1}, {38,1}, {39,1}, {40,1}, {41,1}, {42,1}, {43,1}, {44,2}, {46,1}, {47,2}, {49,1}, {50,1}, {51,2}, {53,1}, {54,1}, {55,2}, {57,1}, {58,1}, {59,2}, {61,1}, {62,2}, {64,1}, {65,1}, {66,1}, {67,0}, {67,0}, {67,1}, {68,1}, {69,1}, {70,2}, {72,1}, {73,1}, {74,1}, {75,1}, {76,1}, {77,1}, {78,1}, {79,2}, {81,2}, {83,1}, {84,2}, {86,2}, {88,1}, {89,1}, {90,1}, {91,1}, {92,1}, {93,1}, {94,1}, {95,2}, {97,2}, {99,1}, {100,2}, {102,0}, {102,1}, {103,1}, {104,1}, {105,1}, {106,1}, {107,1}, {108,1}, {109,1}, {110,1}, {111,1}, {112,1}, {113,1}, {114,1}, {115,1}, {116,1}, {117,1}, {118,2}, {120,1}, {121,1}, {122,1}, {123,1}, {124,1}, {125,1}, {126,1}, {127,2}, {129,1}, {130,1}, {131,1}, {132,1}, {133,1}, {134,0}, {134,0}};
__device__ const float kBVal_w128_l3_collapsed[134] = {
    1.0f, 1.0f, 1.0f, 1.0f, 0.707106769f, 0.707106769f, 0.707106769f, 0.707106769f, -0.408248305f, 0.816496611f, -0.408248305f, 0.707106769f, 0.707106769f, -0.707106769f, 0.707106769f, 0.408248305f, 0.816496611f, -0.408248305f, -0.408248305f, 0.408248305f, -0.707106769f, -0.408248305f, -0.707106769f, 0.707106769f, 0.707106769f, -0.408248305f, -0.408248305f, 0.408248305f, 0.408248305f, -0.816496611f, 0.408248305f, 0.577350259f, 0.577350259f, 0.577350259f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 0.353553385f, 0.866025388f, -0.353553385f, -0.353553385f, 0.456435472f, 0.577350259f, -0.456435472f, -0.353553385f, -0.456435472f, 0.288675129f, -0.707106769f, -0.456435472f, -0.707106769f, 0.707106769f, 0.707106769f, -0.456435472f, -0.288675129f, 0.456435472f, 0.456435472f, -0.353553385f, -0.577350259f, 0.353553385f, 0.456435472f, 0.353553385f, -0.866025388f, 0.353553385f, 1.0f, 1.0f, 1.0f, 0.316227764f, 0.547722578f, -0.547722578f, -0.547722578f, -0.547722578f, -0.632455528f, -0.547722578f, -0.547722578f, -0.547722578f, 0.316227764f, -0.547722578f, 0.154303357f, 0.597614288f, -0.487950027f, -0.597614288f, 0.154303357f, 0.377964467f, 0.487950027f, -0.617213428f, -0.487950027f, -0.534522474f, -0.654653668f, -0.534522474f, -0.487950027f, -0.617213428f, 0.377964467f, -0.487950027f, -0.597614288f, -0.154303357f, -0.487950027f, 0.154303357f, -0.597614288f, 0.707106769f, -0.707106769f, -0.707106769f, 0.707106769f, 0.707106769f, -0.707106769f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 0.707106769f, 0.707106769f, 0.577350259f, 0.577350259f, 0.577350259f, 0.632455528f, 0.182574183f, 0.730296731f, -0.182574183f, -0.44721359f, 0.774596691f, -0.44721359f, -0.182574183f, 0.730296731f, 0.632455528f, -0.182574183f, -0.577350259f, 0.577350259f, 0.577350259f, -0.707106769f, 0.707106769f};
__device__ const unsigned char kBI2_w128_l3_collapsed[134] = {
    0, 1, 2, 3, 3, 1, 2, 1, 1, 2, 3, 3, 2, 1, 3, 5, 8, 7, 4, 7, 6, 8, 7, 5, 6, 8, 5, 4, 7, 4, 5, 1, 2, 3, 9, 10, 11, 12, 13, 14, 15, 10, 15, 14, 9, 11, 14, 13, 15, 10, 13, 12, 14, 13, 11, 12, 14, 11, 10, 13, 15, 10, 9, 11, 14, 9, 10, 0, 0, 0, 6, 8, 5, 4, 5, 6, 7, 4, 7, 6, 8, 13, 15, 10, 9, 11, 12, 14, 11, 10, 11, 12, 13, 10, 13, 12, 14, 9, 11, 14, 13, 15, 3, 2, 3, 1, 2, 1, 4, 5, 6, 7, 8, 8, 4, 7, 4, 5, 6, 8, 5, 4, 5, 6, 7, 4, 7, 6, 8, 5, 8, 7, 4, 8};
__device__ const unsigned char kBRow_w128_l3_collapsed[60] = {
    0, 1, 2, 3, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16, 16, 0, 17, 18, 19, 20, 21, 22, 23, 24, 25, 26, 27, 28, 29, 30, 1, 2, 3, 7, 8, 9, 10, 11, 11, 11, 11, 11, 11, 11, 11, 4, 5, 6, 7, 8, 9, 10, 11, 17, 18, 19, 20, 21, 22, 23};

struct Sig_w128_l3_collapsed {
    static constexpr int NQ = 128, DIN = 4, DSH = 16, P = 13, D = 31;
    static constexpr int NNZ = 134, NPAIR = 116, V = 4;
    static constexpr int FW = 4, FT = 6, FS = 2, FC = 2, F_RMAX = 11, F_APAD = 124, F_NREC = 2, F_NPMAX = 36, F_MAXREG = 255;
    // fused double backward (cotangent of grad_out): tile, stages, CTAs per SM (DFT = 0: not generated)
    static constexpr int DFT = 0, DFS = 2, DFC = 1, DFV = 4;
    using DFVec = float4;
    using Vec = float4;
    __device__ static __forceinline__ PairRec pair_rec(int i) { return kPair_w128_l3_collapsed[i]; }
    __device__ static __forceinline__ float rec_val(int i) { return kVal_w128_l3_collapsed[i]; }
    __device__ static __forceinline__ unsigned char rec_i2(int i) { return kI2_w128_l3_collapsed[i]; }
    static constexpr int f_row0(int g) {
        switch (g) {
            case 0: return 0;
            case 1: return 5;
            case 2: return 11;
            case 3: return 20;
            case 4: return 31;
            default: return 31;
        }
    }
    static constexpr int f_a0(int g) {
        switch (g) {
            case 0: return 0;
            case 1: return 24;
            case 2: return 56;
            case 3: return 88;
            case 4: return 124;
            default: return 124;
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
            pfma(acc[0], a0.y, sx1_1);
            pfma(acc[0], a0.z, sx1_2);
            pfma(acc[0], a0.w, sx1_3);
            const Vec s2 = ss[2 * NQV];  // path 2: l1=0 l2=1 -> L=1
            const Vec sx2_0 = pmul(s2, x0);
            const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
            pfma(acc[1], a1.x, sx2_0);
            const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
            pfma(acc[2], a2.y, sx2_0);
            const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
            pfma(acc[3], a3.z, sx2_0);
            const Vec s3 = ss[3 * NQV];  // path 3: l1=1 l2=0 -> L=1
            const Vec sx3_1 = pmul(s3, x1);
            const Vec sx3_2 = pmul(s3, x2);
            const Vec sx3_3 = pmul(s3, x3);
            pfma(acc[1], a1.y, sx3_1);
            pfma(acc[2], a2.z, sx3_2);
            pfma(acc[3], a3.w, sx3_3);
            const Vec s4 = ss[4 * NQV];  // path 4: l1=1 l2=2 -> L=1
            const Vec sx4_1 = pmul(s4, x1);
            const Vec sx4_2 = pmul(s4, x2);
            const Vec sx4_3 = pmul(s4, x3);
            pfma(acc[1], a1.z, sx4_1);
            pfma(acc[2], a2.w, sx4_1);
            const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
            pfma(acc[3], a4.x, sx4_1);
            pfma(acc[1], a1.w, sx4_2);
            pfma(acc[2], a3.x, sx4_2);
            pfma(acc[3], a4.y, sx4_2);
            pfma(acc[1], a2.x, sx4_3);
            pfma(acc[2], a3.y, sx4_3);
            pfma(acc[3], a4.z, sx4_3);
            const Vec s5 = ss[5 * NQV];  // path 5: l1=1 l2=1 -> L=1
            const Vec sx5_2 = pmul(s5, x2);
            const Vec sx5_3 = pmul(s5, x3);
            pfma(acc[4], a4.w, sx5_2);
            const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
            pfma(acc[4], a5.x, sx5_3);
        }
        if constexpr (G == 1) {
            const Vec x0 = xs[0 * NQV];
            const Vec x1 = xs[1 * NQV];
            const Vec x2 = xs[2 * NQV];
            const Vec x3 = xs[3 * NQV];
            const Vec s5 = ss[5 * NQV];  // path 5: l1=1 l2=1 -> L=1
            const Vec sx5_1 = pmul(s5, x1);
            const Vec sx5_2 = pmul(s5, x2);
            const Vec sx5_3 = pmul(s5, x3);
            const float4 a6 = *reinterpret_cast<const float4*>(As + 24);
            pfma(acc[0], a6.x, sx5_1);
            pfma(acc[1], a6.z, sx5_1);
            pfma(acc[0], a6.y, sx5_3);
            pfma(acc[1], a6.w, sx5_2);
            const Vec s6 = ss[6 * NQV];  // path 6: l1=0 l2=2 -> L=2
            const Vec sx6_0 = pmul(s6, x0);
            const float4 a7 = *reinterpret_cast<const float4*>(As + 28);
            pfma(acc[2], a7.x, sx6_0);
            const float4 a8 = *reinterpret_cast<const float4*>(As + 32);
            pfma(acc[3], a8.z, sx6_0);
            const float4 a10 = *reinterpret_cast<const float4*>(As + 40);
            pfma(acc[4], a10.x, sx6_0);
            const float4 a11 = *reinterpret_cast<const float4*>(As + 44);
            pfma(acc[5], a11.w, sx6_0);
            const Vec s7 = ss[7 * NQV];  // path 7: l1=1 l2=1 -> L=2
            const Vec sx7_1 = pmul(s7, x1);
            const Vec sx7_2 = pmul(s7, x2);
            const Vec sx7_3 = pmul(s7, x3);
            pfma(acc[2], a7.y, sx7_1);
            pfma(acc[3], a8.w, sx7_1);
            pfma(acc[4], a10.y, sx7_1);
            const float4 a12 = *reinterpret_cast<const float4*>(As + 48);
            pfma(acc[5], a12.x, sx7_2);
            pfma(acc[2], a7.z, sx7_3);
            const float4 a9 = *reinterpret_cast<const float4*>(As + 36);
            pfma(acc[3], a9.x, sx7_2);
            pfma(acc[4], a10.z, sx7_2);
            pfma(acc[5], a12.y, sx7_3);
            pfma(acc[4], a10.w, sx7_3);
            const Vec s8 = ss[8 * NQV];  // path 8: l1=1 l2=3 -> L=2
            const Vec sx8_1 = pmul(s8, x1);
            const Vec sx8_2 = pmul(s8, x2);
            const Vec sx8_3 = pmul(s8, x3);
            pfma(acc[2], a7.w, sx8_1);
            pfma(acc[3], a9.y, sx8_1);
            pfma(acc[4], a11.x, sx8_1);
            pfma(acc[5], a12.z, sx8_1);
            pfma(acc[2], a8.x, sx8_2);
            pfma(acc[3], a9.z, sx8_2);
            pfma(acc[4], a11.y, sx8_2);
            pfma(acc[5], a12.w, sx8_2);
            pfma(acc[2], a8.y, sx8_3);
            pfma(acc[3], a9.w, sx8_3);
            pfma(acc[4], a11.z, sx8_3);
            const float4 a13 = *reinterpret_cast<const float4*>(As + 52);
            pfma(acc[5], a13.x, sx8_3);
        }
        if constexpr (G == 2) {
            const Vec x0 = xs[0 * NQV];
            const Vec x1 = xs[1 * NQV];
            const Vec x2 = xs[2 * NQV];
            const Vec x3 = xs[3 * NQV];
            const Vec s6 = ss[6 * NQV];  // path 6: l1=0 l2=2 -> L=2
            const Vec sx6_0 = pmul(s6, x0);
            const float4 a14 = *reinterpret_cast<const float4*>(As + 56);
            pfma(acc[0], a14.x, sx6_0);
            const Vec s7 = ss[7 * NQV];  // path 7: l1=1 l2=1 -> L=2
            const Vec sx7_1 = pmul(s7, x1);
            const Vec sx7_3 = pmul(s7, x3);
            pfma(acc[0], a14.y, sx7_1);
            pfma(acc[0], a14.z, sx7_3);
            const Vec s8 = ss[8 * NQV];  // path 8: l1=1 l2=3 -> L=2
            const Vec sx8_1 = pmul(s8, x1);
            const Vec sx8_2 = pmul(s8, x2);
            const Vec sx8_3 = pmul(s8, x3);
            pfma(acc[0], a14.w, sx8_1);
            const float4 a15 = *reinterpret_cast<const float4*>(As + 60);
            pfma(acc[0], a15.x, sx8_2);
            pfma(acc[0], a15.y, sx8_3);
            const Vec s9 = ss[9 * NQV];  // path 9: l1=1 l2=2 -> L=2
            const Vec sx9_1 = pmul(s9, x1);
            const Vec sx9_2 = pmul(s9, x2);
            const Vec sx9_3 = pmul(s9, x3);
            pfma(acc[1], a15.z, sx9_1);
            const float4 a16 = *reinterpret_cast<const float4*>(As + 64);
            pfma(acc[2], a16.y, sx9_1);
            const float4 a17 = *reinterpret_cast<const float4*>(As + 68);
            pfma(acc[3], a17.x, sx9_1);
            pfma(acc[4], a17.z, sx9_1);
            const float4 a18 = *reinterpret_cast<const float4*>(As + 72);
            pfma(acc[5], a18.y, sx9_1);
            pfma(acc[1], a15.w, sx9_2);
            pfma(acc[2], a16.z, sx9_2);
            pfma(acc[3], a17.y, sx9_3);
            pfma(acc[4], a17.w, sx9_2);
            pfma(acc[5], a18.z, sx9_2);
            pfma(acc[1], a16.x, sx9_3);
            pfma(acc[2], a16.w, sx9_3);
            pfma(acc[4], a18.x, sx9_3);
            pfma(acc[5], a18.w, sx9_3);
            const Vec s10 = ss[10 * NQV];  // path 10: l1=0 l2=3 -> L=3
            const Vec sx10_0 = pmul(s10, x0);
            const float4 a19 = *reinterpret_cast<const float4*>(As + 76);
            pfma(acc[6], a19.x, sx10_0);
            pfma(acc[7], a19.w, sx10_0);
            const float4 a20 = *reinterpret_cast<const float4*>(As + 80);
            pfma(acc[8], a20.w, sx10_0);
            const Vec s11 = ss[11 * NQV];  // path 11: l1=1 l2=2 -> L=3
            const Vec sx11_1 = pmul(s11, x1);
            const Vec sx11_2 = pmul(s11, x2);
            const Vec sx11_3 = pmul(s11, x3);
            pfma(acc[6], a19.y, sx11_1);
            pfma(acc[7], a20.x, sx11_1);
            const float4 a21 = *reinterpret_cast<const float4*>(As + 84);
            pfma(acc[8], a21.x, sx11_1);
            pfma(acc[6], a19.z, sx11_3);
            pfma(acc[7], a20.y, sx11_2);
            pfma(acc[8], a21.y, sx11_2);
            pfma(acc[7], a20.z, sx11_3);
            pfma(acc[8], a21.z, sx11_3);
        }
        if constexpr (G == 3) {
            const Vec x0 = xs[0 * NQV];
            const Vec x1 = xs[1 * NQV];
            const Vec x2 = xs[2 * NQV];
            const Vec x3 = xs[3 * NQV];
            const Vec s10 = ss[10 * NQV];  // path 10: l1=0 l2=3 -> L=3
            const Vec sx10_0 = pmul(s10, x0);
            const float4 a22 = *reinterpret_cast<const float4*>(As + 88);
            pfma(acc[0], a22.x, sx10_0);
            const float4 a23 = *reinterpret_cast<const float4*>(As + 92);
            pfma(acc[1], a23.x, sx10_0);
            const float4 a24 = *reinterpret_cast<const float4*>(As + 96);
            pfma(acc[2], a24.x, sx10_0);
            const float4 a25 = *reinterpret_cast<const float4*>(As + 100);
            pfma(acc[3], a25.x, sx10_0);
            const Vec s11 = ss[11 * NQV];  // path 11: l1=1 l2=2 -> L=3
            const Vec sx11_1 = pmul(s11, x1);
            const Vec sx11_2 = pmul(s11, x2);
            const Vec sx11_3 = pmul(s11, x3);
            pfma(acc[0], a22.y, sx11_1);
            pfma(acc[1], a23.y, sx11_1);
            pfma(acc[2], a24.y, sx11_1);
            pfma(acc[3], a25.y, sx11_1);
            pfma(acc[0], a22.z, sx11_2);
            pfma(acc[1], a23.z, sx11_2);
            pfma(acc[2], a24.z, sx11_2);
            pfma(acc[3], a25.z, sx11_3);
            pfma(acc[0], a22.w, sx11_3);
            pfma(acc[1], a23.w, sx11_3);
            pfma(acc[2], a24.w, sx11_3);
            const Vec s12 = ss[12 * NQV];  // path 12: l1=1 l2=3 -> L=3
            const Vec sx12_1 = pmul(s12, x1);
            const Vec sx12_2 = pmul(s12, x2);
            const Vec sx12_3 = pmul(s12, x3);
            pfma(acc[4], a25.w, sx12_1);
            const float4 a26 = *reinterpret_cast<const float4*>(As + 104);
            pfma(acc[5], a26.z, sx12_1);
            const float4 a27 = *reinterpret_cast<const float4*>(As + 108);
            pfma(acc[6], a27.y, sx12_1);
            const float4 a28 = *reinterpret_cast<const float4*>(As + 112);
            pfma(acc[7], a28.x, sx12_1);
            pfma(acc[8], a28.z, sx12_1);
            const float4 a29 = *reinterpret_cast<const float4*>(As + 116);
            pfma(acc[9], a29.y, sx12_1);
            const float4 a30 = *reinterpret_cast<const float4*>(As + 120);
            pfma(acc[10], a30.x, sx12_1);
            pfma(acc[4], a26.x, sx12_2);
            pfma(acc[5], a26.w, sx12_2);
            pfma(acc[6], a27.z, sx12_2);
            pfma(acc[7], a28.y, sx12_3);
            pfma(acc[8], a28.w, sx12_2);
            pfma(acc[9], a29.z, sx12_2);
            pfma(acc[10], a30.y, sx12_2);
            pfma(acc[4], a26.y, sx12_3);
            pfma(acc[5], a27.x, sx12_3);
            pfma(acc[6], a27.w, sx12_3);
            pfma(acc[8], a29.x, sx12_3);
            pfma(acc[9], a29.w, sx12_3);
            pfma(acc[10], a30.z, sx12_3);
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
        }
        if constexpr (G == 1) {
            dst[0 * stride] = acc[0];
            dst[1 * stride] = acc[1];
            dst[2 * stride] = acc[2];
            dst[3 * stride] = acc[3];
            dst[4 * stride] = acc[4];
            dst[5 * stride] = acc[5];
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
            dst[10 * stride] = acc[10];
        }
    }
    // ---- backward: path groups [[0, 2, 7, 9], [1, 10, 12], [3, 4, 8], [5, 6, 11]]
    static constexpr int BV = 4;  // channels per lane in the backward
    using BVec = float4;
    static constexpr int BW = 4, BT = 5, BS = 2, BC = 2, B_RMAX = 15, B_APAD = 124, B_NREC = 2;
    // edge-wise backward (one warp per edge, grad_out rows read from shared memory): edges per tile (0 = not generated), ring stages
    static constexpr int ET = 7, ES = 2, EV = 4, EXG = 0;   // EXG: sender rows not staged
    static constexpr int ST = 7;   // columns of the scheduled backward
    // the same for the standalone tensor product: rows per ring slot (0 = not generated), ring slots
    static constexpr int ETR = 0, ESR = 3;
    // fused double backward (edge outputs): edges per tile (0 = not generated), ring stages
    static constexpr int DT = 0, DS = 2, DV = 4;
    using DVec = float4;
    using EVec = float4;
    __device__ static __forceinline__ PairRec b_pair_rec(int i) { return kBPair_w128_l3_collapsed[i]; }
    __device__ static __forceinline__ float b_rec_val(int i) { return kBVal_w128_l3_collapsed[i]; }
    __device__ static __forceinline__ unsigned char b_rec_i2(int i) { return kBI2_w128_l3_collapsed[i]; }
    // output rows of path group g: b_nrow(g) of them, the r-th is b_row(g, r)
    __device__ static __forceinline__ int b_row(int g, int r) { return kBRow_w128_l3_collapsed[g * B_RMAX + r]; }
    static constexpr int b_nrow(int g) {
        switch (g) {
            case 0: return 14;
            case 1: return 15;
            case 2: return 8;
            case 3: return 15;
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
            const BVec s2 = ss[2 * NQV];  // path 2: l1=0 l2=1 -> L=1
            const BVec sx2_0 = vmul(s2, x0);
            BVec u2_0; vzero(u2_0);
            vfma(u2_0, a0.y, dm[1]);
            { const float t = vdot(sx2_0, dm[1]);
              dyl[1] = 1.0f * t;
            }
            vfma(u2_0, a0.z, dm[2]);
            { const float t = vdot(sx2_0, dm[2]);
              dyl[2] = 1.0f * t;
            }
            vfma(u2_0, a0.w, dm[3]);
            { const float t = vdot(sx2_0, dm[3]);
              dyl[3] = 1.0f * t;
            }
            BVec ds2 = vmul(x0, u2_0);
            if (gw) gw[2 * NQV] = ds2;
            vfma(dxp[0], s2, u2_0);
            const BVec s7 = ss[7 * NQV];  // path 7: l1=1 l2=1 -> L=2
            const BVec sx7_1 = vmul(s7, x1);
            BVec u7_1; vzero(u7_1);
            const BVec sx7_2 = vmul(s7, x2);
            BVec u7_2; vzero(u7_2);
            const BVec sx7_3 = vmul(s7, x3);
            BVec u7_3; vzero(u7_3);
            const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
            vfma(u7_1, a1.x, dm[4]);
            { const float t = vdot(sx7_1, dm[4]);
              dyl[3] = fmaf(0.707106769f, t, dyl[3]);
            }
            vfma(u7_1, a1.z, dm[5]);
            { const float t = vdot(sx7_1, dm[5]);
              dyl[2] = fmaf(0.707106769f, t, dyl[2]);
            }
            const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
            vfma(u7_1, a2.x, dm[6]);
            { const float t = vdot(sx7_1, dm[6]);
              dyl[1] = fmaf(-0.408248305f, t, dyl[1]);
            }
            vfma(u7_2, a2.w, dm[7]);
            { const float t = vdot(sx7_2, dm[7]);
              dyl[3] = fmaf(0.707106769f, t, dyl[3]);
            }
            const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
            vfma(u7_1, a3.y, dm[8]);
            { const float t = vdot(sx7_1, dm[8]);
              dyl[1] = fmaf(-0.707106769f, t, dyl[1]);
            }
            vfma(u7_3, a1.y, dm[4]);
            { const float t = vdot(sx7_3, dm[4]);
              dyl[1] = fmaf(0.707106769f, t, dyl[1]);
            }
            vfma(u7_2, a1.w, dm[5]);
            { const float t = vdot(sx7_2, dm[5]);
              dyl[1] = fmaf(0.707106769f, t, dyl[1]);
            }
            vfma(u7_2, a2.y, dm[6]);
            { const float t = vdot(sx7_2, dm[6]);
              dyl[2] = fmaf(0.816496611f, t, dyl[2]);
            }
            vfma(u7_3, a3.x, dm[7]);
            { const float t = vdot(sx7_3, dm[7]);
              dyl[2] = fmaf(0.707106769f, t, dyl[2]);
            }
            vfma(u7_3, a3.z, dm[8]);
            { const float t = vdot(sx7_3, dm[8]);
              dyl[3] = fmaf(0.707106769f, t, dyl[3]);
            }
            vfma(u7_3, a2.z, dm[6]);
            { const float t = vdot(sx7_3, dm[6]);
              dyl[3] = fmaf(-0.408248305f, t, dyl[3]);
            }
            BVec ds7 = vmul(x1, u7_1);
            vfma(ds7, x2, u7_2);
            vfma(ds7, x3, u7_3);
            if (gw) gw[7 * NQV] = ds7;
            dxp[1] = vmul(s7, u7_1);
            dxp[2] = vmul(s7, u7_2);
            dxp[3] = vmul(s7, u7_3);
            const BVec s9 = ss[9 * NQV];  // path 9: l1=1 l2=2 -> L=2
            const BVec sx9_1 = vmul(s9, x1);
            BVec u9_1; vzero(u9_1);
            const BVec sx9_2 = vmul(s9, x2);
            BVec u9_2; vzero(u9_2);
            const BVec sx9_3 = vmul(s9, x3);
            BVec u9_3; vzero(u9_3);
            vfma(u9_1, a3.w, dm[9]);
            { const float t = vdot(sx9_1, dm[9]);
              dyl[5] = 0.408248305f * t;
            }
            const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
            vfma(u9_1, a4.z, dm[10]);
            { const float t = vdot(sx9_1, dm[10]);
              dyl[4] = -0.408248305f * t;
            }
            const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
            vfma(u9_1, a5.y, dm[11]);
            { const float t = vdot(sx9_1, dm[11]);
              dyl[7] = -0.707106769f * t;
            }
            vfma(u9_1, a5.w, dm[12]);
            { const float t = vdot(sx9_1, dm[12]);
              dyl[6] = 0.707106769f * t;
              dyl[8] = -0.408248305f * t;
            }
            const float4 a6 = *reinterpret_cast<const float4*>(As + 24);
            vfma(u9_1, a6.z, dm[13]);
            { const float t = vdot(sx9_1, dm[13]);
              dyl[7] = fmaf(0.408248305f, t, dyl[7]);
            }
            vfma(u9_2, a4.x, dm[9]);
            { const float t = vdot(sx9_2, dm[9]);
              dyl[8] = fmaf(0.816496611f, t, dyl[8]);
            }
            vfma(u9_2, a4.w, dm[10]);
            { const float t = vdot(sx9_2, dm[10]);
              dyl[7] = fmaf(0.408248305f, t, dyl[7]);
            }
            vfma(u9_3, a5.z, dm[11]);
            { const float t = vdot(sx9_3, dm[11]);
              dyl[5] = fmaf(0.707106769f, t, dyl[5]);
            }
            vfma(u9_2, a6.x, dm[12]);
            { const float t = vdot(sx9_2, dm[12]);
              dyl[5] = fmaf(-0.408248305f, t, dyl[5]);
            }
            vfma(u9_2, a6.w, dm[13]);
            { const float t = vdot(sx9_2, dm[13]);
              dyl[4] = fmaf(-0.816496611f, t, dyl[4]);
            }
            vfma(u9_3, a4.y, dm[9]);
            { const float t = vdot(sx9_3, dm[9]);
              dyl[7] = fmaf(-0.408248305f, t, dyl[7]);
            }
            vfma(u9_3, a5.x, dm[10]);
            { const float t = vdot(sx9_3, dm[10]);
              dyl[6] = fmaf(-0.707106769f, t, dyl[6]);
              dyl[8] = fmaf(-0.408248305f, t, dyl[8]);
            }
            vfma(u9_3, a6.y, dm[12]);
            { const float t = vdot(sx9_3, dm[12]);
              dyl[4] = fmaf(0.408248305f, t, dyl[4]);
            }
            const float4 a7 = *reinterpret_cast<const float4*>(As + 28);
            vfma(u9_3, a7.x, dm[13]);
            { const float t = vdot(sx9_3, dm[13]);
              dyl[5] = fmaf(0.408248305f, t, dyl[5]);
            }
            BVec ds9 = vmul(x1, u9_1);
            vfma(ds9, x2, u9_2);
            vfma(ds9, x3, u9_3);
            if (gw) gw[9 * NQV] = ds9;
            vfma(dxp[1], s9, u9_1);
            vfma(dxp[2], s9, u9_2);
            vfma(dxp[3], s9, u9_3);
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
            const float4 a8 = *reinterpret_cast<const float4*>(As + 32);
            vfma(u1_1, a8.x, dm[0]);
            { const float t = vdot(sx1_1, dm[0]);
              dyl[1] = 0.577350259f * t;
            }
            vfma(u1_2, a8.y, dm[0]);
            { const float t = vdot(sx1_2, dm[0]);
              dyl[2] = 0.577350259f * t;
            }
            vfma(u1_3, a8.z, dm[0]);
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
            const BVec s10 = ss[10 * NQV];  // path 10: l1=0 l2=3 -> L=3
            const BVec sx10_0 = vmul(s10, x0);
            BVec u10_0; vzero(u10_0);
            vfma(u10_0, a8.w, dm[1]);
            { const float t = vdot(sx10_0, dm[1]);
              dyl[9] = 1.0f * t;
            }
            const float4 a9 = *reinterpret_cast<const float4*>(As + 36);
            vfma(u10_0, a9.x, dm[2]);
            { const float t = vdot(sx10_0, dm[2]);
              dyl[10] = 1.0f * t;
            }
            vfma(u10_0, a9.y, dm[3]);
            { const float t = vdot(sx10_0, dm[3]);
              dyl[11] = 1.0f * t;
            }
            vfma(u10_0, a9.z, dm[4]);
            { const float t = vdot(sx10_0, dm[4]);
              dyl[12] = 1.0f * t;
            }
            vfma(u10_0, a9.w, dm[5]);
            { const float t = vdot(sx10_0, dm[5]);
              dyl[13] = 1.0f * t;
            }
            const float4 a10 = *reinterpret_cast<const float4*>(As + 40);
            vfma(u10_0, a10.x, dm[6]);
            { const float t = vdot(sx10_0, dm[6]);
              dyl[14] = 1.0f * t;
            }
            vfma(u10_0, a10.y, dm[7]);
            { const float t = vdot(sx10_0, dm[7]);
              dyl[15] = 1.0f * t;
            }
            BVec ds10 = vmul(x0, u10_0);
            if (gw) gw[10 * NQV] = ds10;
            dxp[0] = vmul(s10, u10_0);
            const BVec s12 = ss[12 * NQV];  // path 12: l1=1 l2=3 -> L=3
            const BVec sx12_1 = vmul(s12, x1);
            BVec u12_1; vzero(u12_1);
            const BVec sx12_2 = vmul(s12, x2);
            BVec u12_2; vzero(u12_2);
            const BVec sx12_3 = vmul(s12, x3);
            BVec u12_3; vzero(u12_3);
            vfma(u12_1, a10.z, dm[8]);
            { const float t = vdot(sx12_1, dm[8]);
              dyl[10] = fmaf(0.353553385f, t, dyl[10]);
            }
            const float4 a11 = *reinterpret_cast<const float4*>(As + 44);
            vfma(u12_1, a11.y, dm[9]);
            { const float t = vdot(sx12_1, dm[9]);
              dyl[9] = fmaf(-0.353553385f, t, dyl[9]);
              dyl[11] = fmaf(0.456435472f, t, dyl[11]);
            }
            const float4 a12 = *reinterpret_cast<const float4*>(As + 48);
            vfma(u12_1, a12.x, dm[10]);
            { const float t = vdot(sx12_1, dm[10]);
              dyl[10] = fmaf(-0.456435472f, t, dyl[10]);
            }
            vfma(u12_1, a12.w, dm[11]);
            { const float t = vdot(sx12_1, dm[11]);
              dyl[13] = fmaf(-0.707106769f, t, dyl[13]);
            }
            const float4 a13 = *reinterpret_cast<const float4*>(As + 52);
            vfma(u12_1, a13.y, dm[12]);
            { const float t = vdot(sx12_1, dm[12]);
              dyl[12] = fmaf(0.707106769f, t, dyl[12]);
              dyl[14] = fmaf(-0.456435472f, t, dyl[14]);
            }
            const float4 a14 = *reinterpret_cast<const float4*>(As + 56);
            vfma(u12_1, a14.x, dm[13]);
            { const float t = vdot(sx12_1, dm[13]);
              dyl[13] = fmaf(0.456435472f, t, dyl[13]);
              dyl[15] = fmaf(-0.353553385f, t, dyl[15]);
            }
            vfma(u12_1, a14.w, dm[14]);
            { const float t = vdot(sx12_1, dm[14]);
              dyl[14] = fmaf(0.353553385f, t, dyl[14]);
            }
            vfma(u12_2, a10.w, dm[8]);
            { const float t = vdot(sx12_2, dm[8]);
              dyl[15] = fmaf(0.866025388f, t, dyl[15]);
            }
            vfma(u12_2, a11.z, dm[9]);
            { const float t = vdot(sx12_2, dm[9]);
              dyl[14] = fmaf(0.577350259f, t, dyl[14]);
            }
            vfma(u12_2, a12.y, dm[10]);
            { const float t = vdot(sx12_2, dm[10]);
              dyl[13] = fmaf(0.288675129f, t, dyl[13]);
            }
            vfma(u12_3, a13.x, dm[11]);
            { const float t = vdot(sx12_3, dm[11]);
              dyl[11] = fmaf(0.707106769f, t, dyl[11]);
            }
            vfma(u12_2, a13.z, dm[12]);
            { const float t = vdot(sx12_2, dm[12]);
              dyl[11] = fmaf(-0.288675129f, t, dyl[11]);
            }
            vfma(u12_2, a14.y, dm[13]);
            { const float t = vdot(sx12_2, dm[13]);
              dyl[10] = fmaf(-0.577350259f, t, dyl[10]);
            }
            const float4 a15 = *reinterpret_cast<const float4*>(As + 60);
            vfma(u12_2, a15.x, dm[14]);
            { const float t = vdot(sx12_2, dm[14]);
              dyl[9] = fmaf(-0.866025388f, t, dyl[9]);
            }
            vfma(u12_3, a11.x, dm[8]);
            { const float t = vdot(sx12_3, dm[8]);
              dyl[14] = fmaf(-0.353553385f, t, dyl[14]);
            }
            vfma(u12_3, a11.w, dm[9]);
            { const float t = vdot(sx12_3, dm[9]);
              dyl[13] = fmaf(-0.456435472f, t, dyl[13]);
              dyl[15] = fmaf(-0.353553385f, t, dyl[15]);
            }
            vfma(u12_3, a12.z, dm[10]);
            { const float t = vdot(sx12_3, dm[10]);
              dyl[12] = fmaf(-0.707106769f, t, dyl[12]);
              dyl[14] = fmaf(-0.456435472f, t, dyl[14]);
            }
            vfma(u12_3, a13.w, dm[12]);
            { const float t = vdot(sx12_3, dm[12]);
              dyl[10] = fmaf(0.456435472f, t, dyl[10]);
            }
            vfma(u12_3, a14.z, dm[13]);
            { const float t = vdot(sx12_3, dm[13]);
              dyl[9] = fmaf(0.353553385f, t, dyl[9]);
              dyl[11] = fmaf(0.456435472f, t, dyl[11]);
            }
            vfma(u12_3, a15.y, dm[14]);
            { const float t = vdot(sx12_3, dm[14]);
              dyl[10] = fmaf(0.353553385f, t, dyl[10]);
            }
            BVec ds12 = vmul(x1, u12_1);
            vfma(ds12, x2, u12_2);
            vfma(ds12, x3, u12_3);
            if (gw) gw[12 * NQV] = ds12;
            vfma(dxp[1], s12, u12_1);
            vfma(dxp[2], s12, u12_2);
            vfma(dxp[3], s12, u12_3);
            dyl[0] = 0.f;
            dyl[4] = 0.f;
            dyl[5] = 0.f;
            dyl[6] = 0.f;
            dyl[7] = 0.f;
            dyl[8] = 0.f;
        } break;
        case 2: {
            const BVec x1 = xs[1 * NQV];
            const BVec x2 = xs[2 * NQV];
            const BVec x3 = xs[3 * NQV];
            const BVec s3 = ss[3 * NQV];  // path 3: l1=1 l2=0 -> L=1
            const BVec sx3_1 = vmul(s3, x1);
            BVec u3_1; vzero(u3_1);
            const BVec sx3_2 = vmul(s3, x2);
            BVec u3_2; vzero(u3_2);
            const BVec sx3_3 = vmul(s3, x3);
            BVec u3_3; vzero(u3_3);
            const float4 a16 = *reinterpret_cast<const float4*>(As + 64);
            vfma(u3_1, a16.x, dm[0]);
            { const float t = vdot(sx3_1, dm[0]);
              dyl[0] = 1.0f * t;
            }
            vfma(u3_2, a16.y, dm[1]);
            { const float t = vdot(sx3_2, dm[1]);
              dyl[0] = fmaf(1.0f, t, dyl[0]);
            }
            vfma(u3_3, a16.z, dm[2]);
            { const float t = vdot(sx3_3, dm[2]);
              dyl[0] = fmaf(1.0f, t, dyl[0]);
            }
            BVec ds3 = vmul(x1, u3_1);
            vfma(ds3, x2, u3_2);
            vfma(ds3, x3, u3_3);
            if (gw) gw[3 * NQV] = ds3;
            dxp[1] = vmul(s3, u3_1);
            dxp[2] = vmul(s3, u3_2);
            dxp[3] = vmul(s3, u3_3);
            const BVec s4 = ss[4 * NQV];  // path 4: l1=1 l2=2 -> L=1
            const BVec sx4_1 = vmul(s4, x1);
            BVec u4_1; vzero(u4_1);
            const BVec sx4_2 = vmul(s4, x2);
            BVec u4_2; vzero(u4_2);
            const BVec sx4_3 = vmul(s4, x3);
            BVec u4_3; vzero(u4_3);
            vfma(u4_1, a16.w, dm[0]);
            { const float t = vdot(sx4_1, dm[0]);
              dyl[6] = 0.316227764f * t;
              dyl[8] = 0.547722578f * t;
            }
            const float4 a17 = *reinterpret_cast<const float4*>(As + 68);
            vfma(u4_1, a17.z, dm[1]);
            { const float t = vdot(sx4_1, dm[1]);
              dyl[5] = -0.547722578f * t;
            }
            const float4 a18 = *reinterpret_cast<const float4*>(As + 72);
            vfma(u4_1, a18.y, dm[2]);
            { const float t = vdot(sx4_1, dm[2]);
              dyl[4] = -0.547722578f * t;
            }
            vfma(u4_2, a17.x, dm[0]);
            { const float t = vdot(sx4_2, dm[0]);
              dyl[5] = fmaf(-0.547722578f, t, dyl[5]);
            }
            vfma(u4_2, a17.w, dm[1]);
            { const float t = vdot(sx4_2, dm[1]);
              dyl[6] = fmaf(-0.632455528f, t, dyl[6]);
            }
            vfma(u4_2, a18.z, dm[2]);
            { const float t = vdot(sx4_2, dm[2]);
              dyl[7] = -0.547722578f * t;
            }
            vfma(u4_3, a17.y, dm[0]);
            { const float t = vdot(sx4_3, dm[0]);
              dyl[4] = fmaf(-0.547722578f, t, dyl[4]);
            }
            vfma(u4_3, a18.x, dm[1]);
            { const float t = vdot(sx4_3, dm[1]);
              dyl[7] = fmaf(-0.547722578f, t, dyl[7]);
            }
            vfma(u4_3, a18.w, dm[2]);
            { const float t = vdot(sx4_3, dm[2]);
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
            const BVec s8 = ss[8 * NQV];  // path 8: l1=1 l2=3 -> L=2
            const BVec sx8_1 = vmul(s8, x1);
            BVec u8_1; vzero(u8_1);
            const BVec sx8_2 = vmul(s8, x2);
            BVec u8_2; vzero(u8_2);
            const BVec sx8_3 = vmul(s8, x3);
            BVec u8_3; vzero(u8_3);
            const float4 a19 = *reinterpret_cast<const float4*>(As + 76);
            vfma(u8_1, a19.x, dm[3]);
            { const float t = vdot(sx8_1, dm[3]);
              dyl[13] = 0.154303357f * t;
              dyl[15] = 0.597614288f * t;
            }
            vfma(u8_1, a19.w, dm[4]);
            { const float t = vdot(sx8_1, dm[4]);
              dyl[12] = 0.377964467f * t;
              dyl[14] = 0.487950027f * t;
            }
            const float4 a20 = *reinterpret_cast<const float4*>(As + 80);
            vfma(u8_1, a20.z, dm[5]);
            { const float t = vdot(sx8_1, dm[5]);
              dyl[11] = -0.534522474f * t;
            }
            const float4 a21 = *reinterpret_cast<const float4*>(As + 84);
            vfma(u8_1, a21.y, dm[6]);
            { const float t = vdot(sx8_1, dm[6]);
              dyl[10] = -0.487950027f * t;
            }
            const float4 a22 = *reinterpret_cast<const float4*>(As + 88);
            vfma(u8_1, a22.x, dm[7]);
            { const float t = vdot(sx8_1, dm[7]);
              dyl[9] = -0.597614288f * t;
              dyl[11] = fmaf(-0.154303357f, t, dyl[11]);
            }
            vfma(u8_2, a19.y, dm[3]);
            { const float t = vdot(sx8_2, dm[3]);
              dyl[10] = fmaf(-0.487950027f, t, dyl[10]);
            }
            vfma(u8_2, a20.x, dm[4]);
            { const float t = vdot(sx8_2, dm[4]);
              dyl[11] = fmaf(-0.617213428f, t, dyl[11]);
            }
            vfma(u8_2, a20.w, dm[5]);
            { const float t = vdot(sx8_2, dm[5]);
              dyl[12] = fmaf(-0.654653668f, t, dyl[12]);
            }
            vfma(u8_2, a21.z, dm[6]);
            { const float t = vdot(sx8_2, dm[6]);
              dyl[13] = fmaf(-0.617213428f, t, dyl[13]);
            }
            vfma(u8_2, a22.y, dm[7]);
            { const float t = vdot(sx8_2, dm[7]);
              dyl[14] = fmaf(-0.487950027f, t, dyl[14]);
            }
            vfma(u8_3, a19.z, dm[3]);
            { const float t = vdot(sx8_3, dm[3]);
              dyl[9] = fmaf(-0.597614288f, t, dyl[9]);
              dyl[11] = fmaf(0.154303357f, t, dyl[11]);
            }
            vfma(u8_3, a20.y, dm[4]);
            { const float t = vdot(sx8_3, dm[4]);
              dyl[10] = fmaf(-0.487950027f, t, dyl[10]);
            }
            vfma(u8_3, a21.x, dm[5]);
            { const float t = vdot(sx8_3, dm[5]);
              dyl[13] = fmaf(-0.534522474f, t, dyl[13]);
            }
            vfma(u8_3, a21.w, dm[6]);
            { const float t = vdot(sx8_3, dm[6]);
              dyl[12] = fmaf(0.377964467f, t, dyl[12]);
              dyl[14] = fmaf(-0.487950027f, t, dyl[14]);
            }
            vfma(u8_3, a22.z, dm[7]);
            { const float t = vdot(sx8_3, dm[7]);
              dyl[13] = fmaf(0.154303357f, t, dyl[13]);
              dyl[15] = fmaf(-0.597614288f, t, dyl[15]);
            }
            BVec ds8 = vmul(x1, u8_1);
            vfma(ds8, x2, u8_2);
            vfma(ds8, x3, u8_3);
            if (gw) gw[8 * NQV] = ds8;
            vfma(dxp[1], s8, u8_1);
            vfma(dxp[2], s8, u8_2);
            vfma(dxp[3], s8, u8_3);
            vzero(dxp[0]);
            dyl[1] = 0.f;
            dyl[2] = 0.f;
            dyl[3] = 0.f;
        } break;
        case 3: {
            const BVec x0 = xs[0 * NQV];
            const BVec x1 = xs[1 * NQV];
            const BVec x2 = xs[2 * NQV];
            const BVec x3 = xs[3 * NQV];
            const BVec s5 = ss[5 * NQV];  // path 5: l1=1 l2=1 -> L=1
            const BVec sx5_1 = vmul(s5, x1);
            BVec u5_1; vzero(u5_1);
            const BVec sx5_2 = vmul(s5, x2);
            BVec u5_2; vzero(u5_2);
            const BVec sx5_3 = vmul(s5, x3);
            BVec u5_3; vzero(u5_3);
            const float4 a23 = *reinterpret_cast<const float4*>(As + 92);
            vfma(u5_2, a23.x, dm[0]);
            { const float t = vdot(sx5_2, dm[0]);
              dyl[3] = 0.707106769f * t;
            }
            vfma(u5_1, a23.z, dm[1]);
            { const float t = vdot(sx5_1, dm[1]);
              dyl[3] = fmaf(-0.707106769f, t, dyl[3]);
            }
            const float4 a24 = *reinterpret_cast<const float4*>(As + 96);
            vfma(u5_1, a24.x, dm[2]);
            { const float t = vdot(sx5_1, dm[2]);
              dyl[2] = 0.707106769f * t;
            }
            vfma(u5_3, a23.y, dm[0]);
            { const float t = vdot(sx5_3, dm[0]);
              dyl[2] = fmaf(-0.707106769f, t, dyl[2]);
            }
            vfma(u5_3, a23.w, dm[1]);
            { const float t = vdot(sx5_3, dm[1]);
              dyl[1] = 0.707106769f * t;
            }
            vfma(u5_2, a24.y, dm[2]);
            { const float t = vdot(sx5_2, dm[2]);
              dyl[1] = fmaf(-0.707106769f, t, dyl[1]);
            }
            BVec ds5 = vmul(x1, u5_1);
            vfma(ds5, x2, u5_2);
            vfma(ds5, x3, u5_3);
            if (gw) gw[5 * NQV] = ds5;
            dxp[1] = vmul(s5, u5_1);
            dxp[2] = vmul(s5, u5_2);
            dxp[3] = vmul(s5, u5_3);
            const BVec s6 = ss[6 * NQV];  // path 6: l1=0 l2=2 -> L=2
            const BVec sx6_0 = vmul(s6, x0);
            BVec u6_0; vzero(u6_0);
            vfma(u6_0, a24.z, dm[3]);
            { const float t = vdot(sx6_0, dm[3]);
              dyl[4] = 1.0f * t;
            }
            vfma(u6_0, a24.w, dm[4]);
            { const float t = vdot(sx6_0, dm[4]);
              dyl[5] = 1.0f * t;
            }
            const float4 a25 = *reinterpret_cast<const float4*>(As + 100);
            vfma(u6_0, a25.x, dm[5]);
            { const float t = vdot(sx6_0, dm[5]);
              dyl[6] = 1.0f * t;
            }
            vfma(u6_0, a25.y, dm[6]);
            { const float t = vdot(sx6_0, dm[6]);
              dyl[7] = 1.0f * t;
            }
            vfma(u6_0, a25.z, dm[7]);
            { const float t = vdot(sx6_0, dm[7]);
              dyl[8] = 1.0f * t;
            }
            BVec ds6 = vmul(x0, u6_0);
            if (gw) gw[6 * NQV] = ds6;
            dxp[0] = vmul(s6, u6_0);
            const BVec s11 = ss[11 * NQV];  // path 11: l1=1 l2=2 -> L=3
            const BVec sx11_1 = vmul(s11, x1);
            BVec u11_1; vzero(u11_1);
            const BVec sx11_2 = vmul(s11, x2);
            BVec u11_2; vzero(u11_2);
            const BVec sx11_3 = vmul(s11, x3);
            BVec u11_3; vzero(u11_3);
            vfma(u11_1, a25.w, dm[8]);
            { const float t = vdot(sx11_1, dm[8]);
              dyl[8] = fmaf(0.707106769f, t, dyl[8]);
            }
            const float4 a26 = *reinterpret_cast<const float4*>(As + 104);
            vfma(u11_1, a26.y, dm[9]);
            { const float t = vdot(sx11_1, dm[9]);
              dyl[7] = fmaf(0.577350259f, t, dyl[7]);
            }
            const float4 a27 = *reinterpret_cast<const float4*>(As + 108);
            vfma(u11_1, a27.x, dm[10]);
            { const float t = vdot(sx11_1, dm[10]);
              dyl[6] = fmaf(0.632455528f, t, dyl[6]);
              dyl[8] = fmaf(0.182574183f, t, dyl[8]);
            }
            vfma(u11_1, a27.w, dm[11]);
            { const float t = vdot(sx11_1, dm[11]);
              dyl[5] = fmaf(-0.44721359f, t, dyl[5]);
            }
            const float4 a28 = *reinterpret_cast<const float4*>(As + 112);
            vfma(u11_1, a28.z, dm[12]);
            { const float t = vdot(sx11_1, dm[12]);
              dyl[4] = fmaf(-0.182574183f, t, dyl[4]);
            }
            const float4 a29 = *reinterpret_cast<const float4*>(As + 116);
            vfma(u11_1, a29.y, dm[13]);
            { const float t = vdot(sx11_1, dm[13]);
              dyl[5] = fmaf(-0.577350259f, t, dyl[5]);
            }
            const float4 a30 = *reinterpret_cast<const float4*>(As + 120);
            vfma(u11_1, a30.x, dm[14]);
            { const float t = vdot(sx11_1, dm[14]);
              dyl[4] = fmaf(-0.707106769f, t, dyl[4]);
            }
            vfma(u11_3, a26.x, dm[8]);
            { const float t = vdot(sx11_3, dm[8]);
              dyl[4] = fmaf(0.707106769f, t, dyl[4]);
            }
            vfma(u11_2, a26.z, dm[9]);
            { const float t = vdot(sx11_2, dm[9]);
              dyl[4] = fmaf(0.577350259f, t, dyl[4]);
            }
            vfma(u11_2, a27.y, dm[10]);
            { const float t = vdot(sx11_2, dm[10]);
              dyl[5] = fmaf(0.730296731f, t, dyl[5]);
            }
            vfma(u11_2, a28.x, dm[11]);
            { const float t = vdot(sx11_2, dm[11]);
              dyl[6] = fmaf(0.774596691f, t, dyl[6]);
            }
            vfma(u11_2, a28.w, dm[12]);
            { const float t = vdot(sx11_2, dm[12]);
              dyl[7] = fmaf(0.730296731f, t, dyl[7]);
            }
            vfma(u11_2, a29.z, dm[13]);
            { const float t = vdot(sx11_2, dm[13]);
              dyl[8] = fmaf(0.577350259f, t, dyl[8]);
            }
            vfma(u11_3, a30.y, dm[14]);
            { const float t = vdot(sx11_3, dm[14]);
              dyl[8] = fmaf(0.707106769f, t, dyl[8]);
            }
            vfma(u11_3, a26.w, dm[9]);
            { const float t = vdot(sx11_3, dm[9]);
              dyl[5] = fmaf(0.577350259f, t, dyl[5]);
            }
            vfma(u11_3, a27.z, dm[10]);
            { const float t = vdot(sx11_3, dm[10]);
              dyl[4] = fmaf(-0.182574183f, t, dyl[4]);
            }
            vfma(u11_3, a28.y, dm[11]);
            { const float t = vdot(sx11_3, dm[11]);
              dyl[7] = fmaf(-0.44721359f, t, dyl[7]);
            }
            vfma(u11_3, a29.x, dm[12]);
            { const float t = vdot(sx11_3, dm[12]);
              dyl[6] = fmaf(0.632455528f, t, dyl[6]);
              dyl[8] = fmaf(-0.182574183f, t, dyl[8]);
            }
            vfma(u11_3, a29.w, dm[13]);
            { const float t = vdot(sx11_3, dm[13]);
              dyl[7] = fmaf(0.577350259f, t, dyl[7]);
            }
            BVec ds11 = vmul(x1, u11_1);
            vfma(ds11, x2, u11_2);
            vfma(ds11, x3, u11_3);
            if (gw) gw[11 * NQV] = ds11;
            vfma(dxp[1], s11, u11_1);
            vfma(dxp[2], s11, u11_2);
            vfma(dxp[3], s11, u11_3);
            dyl[0] = 0.f;
            dyl[9] = 0.f;
            dyl[10] = 0.f;
            dyl[11] = 0.f;
            dyl[12] = 0.f;
            dyl[13] = 0.f;
            dyl[14] = 0.f;
            dyl[15] = 0.f;
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
        const EVec d1_0 = dms[0 * NQV];
        const float4 a8 = *reinterpret_cast<const float4*>(As + 32);
        vfma(u1_1, a8.x, d1_0);
        { const float t = vdot(sx1_1, d1_0);
          dyl[1] = 0.577350259f * t;
        }
        vfma(u1_2, a8.y, d1_0);
        { const float t = vdot(sx1_2, d1_0);
          dyl[2] = 0.577350259f * t;
        }
        vfma(u1_3, a8.z, d1_0);
        { const float t = vdot(sx1_3, d1_0);
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
        const EVec d2_1 = dms[1 * NQV];
        vfma(u2_0, a0.y, d2_1);
        { const float t = vdot(sx2_0, d2_1);
          dyl[1] = fmaf(1.0f, t, dyl[1]);
        }
        const EVec d2_2 = dms[2 * NQV];
        vfma(u2_0, a0.z, d2_2);
        { const float t = vdot(sx2_0, d2_2);
          dyl[2] = fmaf(1.0f, t, dyl[2]);
        }
        const EVec d2_3 = dms[3 * NQV];
        vfma(u2_0, a0.w, d2_3);
        { const float t = vdot(sx2_0, d2_3);
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
        const EVec d3_1 = dms[1 * NQV];
        const float4 a16 = *reinterpret_cast<const float4*>(As + 64);
        vfma(u3_1, a16.x, d3_1);
        { const float t = vdot(sx3_1, d3_1);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        const EVec d3_2 = dms[2 * NQV];
        vfma(u3_2, a16.y, d3_2);
        { const float t = vdot(sx3_2, d3_2);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        const EVec d3_3 = dms[3 * NQV];
        vfma(u3_3, a16.z, d3_3);
        { const float t = vdot(sx3_3, d3_3);
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
        const EVec d4_1 = dms[1 * NQV];
        vfma(u4_1, a16.w, d4_1);
        { const float t = vdot(sx4_1, d4_1);
          dyl[6] = 0.316227764f * t;
          dyl[8] = 0.547722578f * t;
        }
        const EVec d4_2 = dms[2 * NQV];
        const float4 a17 = *reinterpret_cast<const float4*>(As + 68);
        vfma(u4_1, a17.z, d4_2);
        { const float t = vdot(sx4_1, d4_2);
          dyl[5] = -0.547722578f * t;
        }
        const EVec d4_3 = dms[3 * NQV];
        const float4 a18 = *reinterpret_cast<const float4*>(As + 72);
        vfma(u4_1, a18.y, d4_3);
        { const float t = vdot(sx4_1, d4_3);
          dyl[4] = -0.547722578f * t;
        }
        vfma(u4_2, a17.x, d4_1);
        { const float t = vdot(sx4_2, d4_1);
          dyl[5] = fmaf(-0.547722578f, t, dyl[5]);
        }
        vfma(u4_2, a17.w, d4_2);
        { const float t = vdot(sx4_2, d4_2);
          dyl[6] = fmaf(-0.632455528f, t, dyl[6]);
        }
        vfma(u4_2, a18.z, d4_3);
        { const float t = vdot(sx4_2, d4_3);
          dyl[7] = -0.547722578f * t;
        }
        vfma(u4_3, a17.y, d4_1);
        { const float t = vdot(sx4_3, d4_1);
          dyl[4] = fmaf(-0.547722578f, t, dyl[4]);
        }
        vfma(u4_3, a18.x, d4_2);
        { const float t = vdot(sx4_3, d4_2);
          dyl[7] = fmaf(-0.547722578f, t, dyl[7]);
        }
        vfma(u4_3, a18.w, d4_3);
        { const float t = vdot(sx4_3, d4_3);
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
        const EVec s5 = ss[5 * NQV];  // path 5: l1=1 l2=1 -> L=1
        const EVec sx5_1 = vmul(s5, x1);
        EVec u5_1; vzero(u5_1);
        const EVec sx5_2 = vmul(s5, x2);
        EVec u5_2; vzero(u5_2);
        const EVec sx5_3 = vmul(s5, x3);
        EVec u5_3; vzero(u5_3);
        const EVec d5_4 = dms[4 * NQV];
        const float4 a23 = *reinterpret_cast<const float4*>(As + 92);
        vfma(u5_2, a23.x, d5_4);
        { const float t = vdot(sx5_2, d5_4);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        const EVec d5_5 = dms[5 * NQV];
        vfma(u5_1, a23.z, d5_5);
        { const float t = vdot(sx5_1, d5_5);
          dyl[3] = fmaf(-0.707106769f, t, dyl[3]);
        }
        const EVec d5_6 = dms[6 * NQV];
        const float4 a24 = *reinterpret_cast<const float4*>(As + 96);
        vfma(u5_1, a24.x, d5_6);
        { const float t = vdot(sx5_1, d5_6);
          dyl[2] = fmaf(0.707106769f, t, dyl[2]);
        }
        vfma(u5_3, a23.y, d5_4);
        { const float t = vdot(sx5_3, d5_4);
          dyl[2] = fmaf(-0.707106769f, t, dyl[2]);
        }
        vfma(u5_3, a23.w, d5_5);
        { const float t = vdot(sx5_3, d5_5);
          dyl[1] = fmaf(0.707106769f, t, dyl[1]);
        }
        vfma(u5_2, a24.y, d5_6);
        { const float t = vdot(sx5_2, d5_6);
          dyl[1] = fmaf(-0.707106769f, t, dyl[1]);
        }
        EVec ds5 = vmul(x1, u5_1);
        vfma(ds5, x2, u5_2);
        vfma(ds5, x3, u5_3);
        if (gw) gw[5 * NQV] = ds5;
        vfma(dxp[1], s5, u5_1);
        vfma(dxp[2], s5, u5_2);
        vfma(dxp[3], s5, u5_3);
        const EVec s6 = ss[6 * NQV];  // path 6: l1=0 l2=2 -> L=2
        const EVec sx6_0 = vmul(s6, x0);
        EVec u6_0; vzero(u6_0);
        const EVec d6_7 = dms[7 * NQV];
        vfma(u6_0, a24.z, d6_7);
        { const float t = vdot(sx6_0, d6_7);
          dyl[4] = fmaf(1.0f, t, dyl[4]);
        }
        const EVec d6_8 = dms[8 * NQV];
        vfma(u6_0, a24.w, d6_8);
        { const float t = vdot(sx6_0, d6_8);
          dyl[5] = fmaf(1.0f, t, dyl[5]);
        }
        const EVec d6_9 = dms[9 * NQV];
        const float4 a25 = *reinterpret_cast<const float4*>(As + 100);
        vfma(u6_0, a25.x, d6_9);
        { const float t = vdot(sx6_0, d6_9);
          dyl[6] = fmaf(1.0f, t, dyl[6]);
        }
        const EVec d6_10 = dms[10 * NQV];
        vfma(u6_0, a25.y, d6_10);
        { const float t = vdot(sx6_0, d6_10);
          dyl[7] = fmaf(1.0f, t, dyl[7]);
        }
        const EVec d6_11 = dms[11 * NQV];
        vfma(u6_0, a25.z, d6_11);
        { const float t = vdot(sx6_0, d6_11);
          dyl[8] = fmaf(1.0f, t, dyl[8]);
        }
        EVec ds6 = vmul(x0, u6_0);
        if (gw) gw[6 * NQV] = ds6;
        vfma(dxp[0], s6, u6_0);
        const EVec s7 = ss[7 * NQV];  // path 7: l1=1 l2=1 -> L=2
        const EVec sx7_1 = vmul(s7, x1);
        EVec u7_1; vzero(u7_1);
        const EVec sx7_2 = vmul(s7, x2);
        EVec u7_2; vzero(u7_2);
        const EVec sx7_3 = vmul(s7, x3);
        EVec u7_3; vzero(u7_3);
        const EVec d7_7 = dms[7 * NQV];
        const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
        vfma(u7_1, a1.x, d7_7);
        { const float t = vdot(sx7_1, d7_7);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        const EVec d7_8 = dms[8 * NQV];
        vfma(u7_1, a1.z, d7_8);
        { const float t = vdot(sx7_1, d7_8);
          dyl[2] = fmaf(0.707106769f, t, dyl[2]);
        }
        const EVec d7_9 = dms[9 * NQV];
        const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
        vfma(u7_1, a2.x, d7_9);
        { const float t = vdot(sx7_1, d7_9);
          dyl[1] = fmaf(-0.408248305f, t, dyl[1]);
        }
        const EVec d7_10 = dms[10 * NQV];
        vfma(u7_2, a2.w, d7_10);
        { const float t = vdot(sx7_2, d7_10);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        const EVec d7_11 = dms[11 * NQV];
        const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
        vfma(u7_1, a3.y, d7_11);
        { const float t = vdot(sx7_1, d7_11);
          dyl[1] = fmaf(-0.707106769f, t, dyl[1]);
        }
        vfma(u7_3, a1.y, d7_7);
        { const float t = vdot(sx7_3, d7_7);
          dyl[1] = fmaf(0.707106769f, t, dyl[1]);
        }
        vfma(u7_2, a1.w, d7_8);
        { const float t = vdot(sx7_2, d7_8);
          dyl[1] = fmaf(0.707106769f, t, dyl[1]);
        }
        vfma(u7_2, a2.y, d7_9);
        { const float t = vdot(sx7_2, d7_9);
          dyl[2] = fmaf(0.816496611f, t, dyl[2]);
        }
        vfma(u7_3, a3.x, d7_10);
        { const float t = vdot(sx7_3, d7_10);
          dyl[2] = fmaf(0.707106769f, t, dyl[2]);
        }
        vfma(u7_3, a3.z, d7_11);
        { const float t = vdot(sx7_3, d7_11);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        vfma(u7_3, a2.z, d7_9);
        { const float t = vdot(sx7_3, d7_9);
          dyl[3] = fmaf(-0.408248305f, t, dyl[3]);
        }
        EVec ds7 = vmul(x1, u7_1);
        vfma(ds7, x2, u7_2);
        vfma(ds7, x3, u7_3);
        if (gw) gw[7 * NQV] = ds7;
        vfma(dxp[1], s7, u7_1);
        vfma(dxp[2], s7, u7_2);
        vfma(dxp[3], s7, u7_3);
        const EVec s8 = ss[8 * NQV];  // path 8: l1=1 l2=3 -> L=2
        const EVec sx8_1 = vmul(s8, x1);
        EVec u8_1; vzero(u8_1);
        const EVec sx8_2 = vmul(s8, x2);
        EVec u8_2; vzero(u8_2);
        const EVec sx8_3 = vmul(s8, x3);
        EVec u8_3; vzero(u8_3);
        const EVec d8_7 = dms[7 * NQV];
        const float4 a19 = *reinterpret_cast<const float4*>(As + 76);
        vfma(u8_1, a19.x, d8_7);
        { const float t = vdot(sx8_1, d8_7);
          dyl[13] = 0.154303357f * t;
          dyl[15] = 0.597614288f * t;
        }
        const EVec d8_8 = dms[8 * NQV];
        vfma(u8_1, a19.w, d8_8);
        { const float t = vdot(sx8_1, d8_8);
          dyl[12] = 0.377964467f * t;
          dyl[14] = 0.487950027f * t;
        }
        const EVec d8_9 = dms[9 * NQV];
        const float4 a20 = *reinterpret_cast<const float4*>(As + 80);
        vfma(u8_1, a20.z, d8_9);
        { const float t = vdot(sx8_1, d8_9);
          dyl[11] = -0.534522474f * t;
        }
        const EVec d8_10 = dms[10 * NQV];
        const float4 a21 = *reinterpret_cast<const float4*>(As + 84);
        vfma(u8_1, a21.y, d8_10);
        { const float t = vdot(sx8_1, d8_10);
          dyl[10] = -0.487950027f * t;
        }
        const EVec d8_11 = dms[11 * NQV];
        const float4 a22 = *reinterpret_cast<const float4*>(As + 88);
        vfma(u8_1, a22.x, d8_11);
        { const float t = vdot(sx8_1, d8_11);
          dyl[9] = -0.597614288f * t;
          dyl[11] = fmaf(-0.154303357f, t, dyl[11]);
        }
        vfma(u8_2, a19.y, d8_7);
        { const float t = vdot(sx8_2, d8_7);
          dyl[10] = fmaf(-0.487950027f, t, dyl[10]);
        }
        vfma(u8_2, a20.x, d8_8);
        { const float t = vdot(sx8_2, d8_8);
          dyl[11] = fmaf(-0.617213428f, t, dyl[11]);
        }
        vfma(u8_2, a20.w, d8_9);
        { const float t = vdot(sx8_2, d8_9);
          dyl[12] = fmaf(-0.654653668f, t, dyl[12]);
        }
        vfma(u8_2, a21.z, d8_10);
        { const float t = vdot(sx8_2, d8_10);
          dyl[13] = fmaf(-0.617213428f, t, dyl[13]);
        }
        vfma(u8_2, a22.y, d8_11);
        { const float t = vdot(sx8_2, d8_11);
          dyl[14] = fmaf(-0.487950027f, t, dyl[14]);
        }
        vfma(u8_3, a19.z, d8_7);
        { const float t = vdot(sx8_3, d8_7);
          dyl[9] = fmaf(-0.597614288f, t, dyl[9]);
          dyl[11] = fmaf(0.154303357f, t, dyl[11]);
        }
        vfma(u8_3, a20.y, d8_8);
        { const float t = vdot(sx8_3, d8_8);
          dyl[10] = fmaf(-0.487950027f, t, dyl[10]);
        }
        vfma(u8_3, a21.x, d8_9);
        { const float t = vdot(sx8_3, d8_9);
          dyl[13] = fmaf(-0.534522474f, t, dyl[13]);
        }
        vfma(u8_3, a21.w, d8_10);
        { const float t = vdot(sx8_3, d8_10);
          dyl[12] = fmaf(0.377964467f, t, dyl[12]);
          dyl[14] = fmaf(-0.487950027f, t, dyl[14]);
        }
        vfma(u8_3, a22.z, d8_11);
        { const float t = vdot(sx8_3, d8_11);
          dyl[13] = fmaf(0.154303357f, t, dyl[13]);
          dyl[15] = fmaf(-0.597614288f, t, dyl[15]);
        }
        EVec ds8 = vmul(x1, u8_1);
        vfma(ds8, x2, u8_2);
        vfma(ds8, x3, u8_3);
        if (gw) gw[8 * NQV] = ds8;
        vfma(dxp[1], s8, u8_1);
        vfma(dxp[2], s8, u8_2);
        vfma(dxp[3], s8, u8_3);
        const EVec s9 = ss[9 * NQV];  // path 9: l1=1 l2=2 -> L=2
        const EVec sx9_1 = vmul(s9, x1);
        EVec u9_1; vzero(u9_1);
        const EVec sx9_2 = vmul(s9, x2);
        EVec u9_2; vzero(u9_2);
        const EVec sx9_3 = vmul(s9, x3);
        EVec u9_3; vzero(u9_3);
        const EVec d9_12 = dms[12 * NQV];
        vfma(u9_1, a3.w, d9_12);
        { const float t = vdot(sx9_1, d9_12);
          dyl[5] = fmaf(0.408248305f, t, dyl[5]);
        }
        const EVec d9_13 = dms[13 * NQV];
        const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
        vfma(u9_1, a4.z, d9_13);
        { const float t = vdot(sx9_1, d9_13);
          dyl[4] = fmaf(-0.408248305f, t, dyl[4]);
        }
        const EVec d9_14 = dms[14 * NQV];
        const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
        vfma(u9_1, a5.y, d9_14);
        { const float t = vdot(sx9_1, d9_14);
          dyl[7] = fmaf(-0.707106769f, t, dyl[7]);
        }
        const EVec d9_15 = dms[15 * NQV];
        vfma(u9_1, a5.w, d9_15);
        { const float t = vdot(sx9_1, d9_15);
          dyl[6] = fmaf(0.707106769f, t, dyl[6]);
          dyl[8] = fmaf(-0.408248305f, t, dyl[8]);
        }
        const EVec d9_16 = dms[16 * NQV];
        const float4 a6 = *reinterpret_cast<const float4*>(As + 24);
        vfma(u9_1, a6.z, d9_16);
        { const float t = vdot(sx9_1, d9_16);
          dyl[7] = fmaf(0.408248305f, t, dyl[7]);
        }
        vfma(u9_2, a4.x, d9_12);
        { const float t = vdot(sx9_2, d9_12);
          dyl[8] = fmaf(0.816496611f, t, dyl[8]);
        }
        vfma(u9_2, a4.w, d9_13);
        { const float t = vdot(sx9_2, d9_13);
          dyl[7] = fmaf(0.408248305f, t, dyl[7]);
        }
        vfma(u9_3, a5.z, d9_14);
        { const float t = vdot(sx9_3, d9_14);
          dyl[5] = fmaf(0.707106769f, t, dyl[5]);
        }
        vfma(u9_2, a6.x, d9_15);
        { const float t = vdot(sx9_2, d9_15);
          dyl[5] = fmaf(-0.408248305f, t, dyl[5]);
        }
        vfma(u9_2, a6.w, d9_16);
        { const float t = vdot(sx9_2, d9_16);
          dyl[4] = fmaf(-0.816496611f, t, dyl[4]);
        }
        vfma(u9_3, a4.y, d9_12);
        { const float t = vdot(sx9_3, d9_12);
          dyl[7] = fmaf(-0.408248305f, t, dyl[7]);
        }
        vfma(u9_3, a5.x, d9_13);
        { const float t = vdot(sx9_3, d9_13);
          dyl[6] = fmaf(-0.707106769f, t, dyl[6]);
          dyl[8] = fmaf(-0.408248305f, t, dyl[8]);
        }
        vfma(u9_3, a6.y, d9_15);
        { const float t = vdot(sx9_3, d9_15);
          dyl[4] = fmaf(0.408248305f, t, dyl[4]);
        }
        const float4 a7 = *reinterpret_cast<const float4*>(As + 28);
        vfma(u9_3, a7.x, d9_16);
        { const float t = vdot(sx9_3, d9_16);
          dyl[5] = fmaf(0.408248305f, t, dyl[5]);
        }
        EVec ds9 = vmul(x1, u9_1);
        vfma(ds9, x2, u9_2);
        vfma(ds9, x3, u9_3);
        if (gw) gw[9 * NQV] = ds9;
        vfma(dxp[1], s9, u9_1);
        vfma(dxp[2], s9, u9_2);
        vfma(dxp[3], s9, u9_3);
        const EVec s10 = ss[10 * NQV];  // path 10: l1=0 l2=3 -> L=3
        const EVec sx10_0 = vmul(s10, x0);
        EVec u10_0; vzero(u10_0);
        const EVec d10_17 = dms[17 * NQV];
        vfma(u10_0, a8.w, d10_17);
        { const float t = vdot(sx10_0, d10_17);
          dyl[9] = fmaf(1.0f, t, dyl[9]);
        }
        const EVec d10_18 = dms[18 * NQV];
        const float4 a9 = *reinterpret_cast<const float4*>(As + 36);
        vfma(u10_0, a9.x, d10_18);
        { const float t = vdot(sx10_0, d10_18);
          dyl[10] = fmaf(1.0f, t, dyl[10]);
        }
        const EVec d10_19 = dms[19 * NQV];
        vfma(u10_0, a9.y, d10_19);
        { const float t = vdot(sx10_0, d10_19);
          dyl[11] = fmaf(1.0f, t, dyl[11]);
        }
        const EVec d10_20 = dms[20 * NQV];
        vfma(u10_0, a9.z, d10_20);
        { const float t = vdot(sx10_0, d10_20);
          dyl[12] = fmaf(1.0f, t, dyl[12]);
        }
        const EVec d10_21 = dms[21 * NQV];
        vfma(u10_0, a9.w, d10_21);
        { const float t = vdot(sx10_0, d10_21);
          dyl[13] = fmaf(1.0f, t, dyl[13]);
        }
        const EVec d10_22 = dms[22 * NQV];
        const float4 a10 = *reinterpret_cast<const float4*>(As + 40);
        vfma(u10_0, a10.x, d10_22);
        { const float t = vdot(sx10_0, d10_22);
          dyl[14] = fmaf(1.0f, t, dyl[14]);
        }
        const EVec d10_23 = dms[23 * NQV];
        vfma(u10_0, a10.y, d10_23);
        { const float t = vdot(sx10_0, d10_23);
          dyl[15] = fmaf(1.0f, t, dyl[15]);
        }
        EVec ds10 = vmul(x0, u10_0);
        if (gw) gw[10 * NQV] = ds10;
        vfma(dxp[0], s10, u10_0);
        const EVec s11 = ss[11 * NQV];  // path 11: l1=1 l2=2 -> L=3
        const EVec sx11_1 = vmul(s11, x1);
        EVec u11_1; vzero(u11_1);
        const EVec sx11_2 = vmul(s11, x2);
        EVec u11_2; vzero(u11_2);
        const EVec sx11_3 = vmul(s11, x3);
        EVec u11_3; vzero(u11_3);
        const EVec d11_17 = dms[17 * NQV];
        vfma(u11_1, a25.w, d11_17);
        { const float t = vdot(sx11_1, d11_17);
          dyl[8] = fmaf(0.707106769f, t, dyl[8]);
        }
        const EVec d11_18 = dms[18 * NQV];
        const float4 a26 = *reinterpret_cast<const float4*>(As + 104);
        vfma(u11_1, a26.y, d11_18);
        { const float t = vdot(sx11_1, d11_18);
          dyl[7] = fmaf(0.577350259f, t, dyl[7]);
        }
        const EVec d11_19 = dms[19 * NQV];
        const float4 a27 = *reinterpret_cast<const float4*>(As + 108);
        vfma(u11_1, a27.x, d11_19);
        { const float t = vdot(sx11_1, d11_19);
          dyl[6] = fmaf(0.632455528f, t, dyl[6]);
          dyl[8] = fmaf(0.182574183f, t, dyl[8]);
        }
        const EVec d11_20 = dms[20 * NQV];
        vfma(u11_1, a27.w, d11_20);
        { const float t = vdot(sx11_1, d11_20);
          dyl[5] = fmaf(-0.44721359f, t, dyl[5]);
        }
        const EVec d11_21 = dms[21 * NQV];
        const float4 a28 = *reinterpret_cast<const float4*>(As + 112);
        vfma(u11_1, a28.z, d11_21);
        { const float t = vdot(sx11_1, d11_21);
          dyl[4] = fmaf(-0.182574183f, t, dyl[4]);
        }
        const EVec d11_22 = dms[22 * NQV];
        const float4 a29 = *reinterpret_cast<const float4*>(As + 116);
        vfma(u11_1, a29.y, d11_22);
        { const float t = vdot(sx11_1, d11_22);
          dyl[5] = fmaf(-0.577350259f, t, dyl[5]);
        }
        const EVec d11_23 = dms[23 * NQV];
        const float4 a30 = *reinterpret_cast<const float4*>(As + 120);
        vfma(u11_1, a30.x, d11_23);
        { const float t = vdot(sx11_1, d11_23);
          dyl[4] = fmaf(-0.707106769f, t, dyl[4]);
        }
        vfma(u11_3, a26.x, d11_17);
        { const float t = vdot(sx11_3, d11_17);
          dyl[4] = fmaf(0.707106769f, t, dyl[4]);
        }
        vfma(u11_2, a26.z, d11_18);
        { const float t = vdot(sx11_2, d11_18);
          dyl[4] = fmaf(0.577350259f, t, dyl[4]);
        }
        vfma(u11_2, a27.y, d11_19);
        { const float t = vdot(sx11_2, d11_19);
          dyl[5] = fmaf(0.730296731f, t, dyl[5]);
        }
        vfma(u11_2, a28.x, d11_20);
        { const float t = vdot(sx11_2, d11_20);
          dyl[6] = fmaf(0.774596691f, t, dyl[6]);
        }
        vfma(u11_2, a28.w, d11_21);
        { const float t = vdot(sx11_2, d11_21);
          dyl[7] = fmaf(0.730296731f, t, dyl[7]);
        }
        vfma(u11_2, a29.z, d11_22);
        { const float t = vdot(sx11_2, d11_22);
          dyl[8] = fmaf(0.577350259f, t, dyl[8]);
        }
        vfma(u11_3, a30.y, d11_23);
        { const float t = vdot(sx11_3, d11_23);
          dyl[8] = fmaf(0.707106769f, t, dyl[8]);
        }
        vfma(u11_3, a26.w, d11_18);
        { const float t = vdot(sx11_3, d11_18);
          dyl[5] = fmaf(0.577350259f, t, dyl[5]);
        }
        vfma(u11_3, a27.z, d11_19);
        { const float t = vdot(sx11_3, d11_19);
          dyl[4] = fmaf(-0.182574183f, t, dyl[4]);
        }
        vfma(u11_3, a28.y, d11_20);
        { const float t = vdot(sx11_3, d11_20);
          dyl[7] = fmaf(-0.44721359f, t, dyl[7]);
        }
        vfma(u11_3, a29.x, d11_21);
        { const float t = vdot(sx11_3, d11_21);
          dyl[6] = fmaf(0.632455528f, t, dyl[6]);
          dyl[8] = fmaf(-0.182574183f, t, dyl[8]);
        }
        vfma(u11_3, a29.w, d11_22);
        { const float t = vdot(sx11_3, d11_22);
          dyl[7] = fmaf(0.577350259f, t, dyl[7]);
        }
        EVec ds11 = vmul(x1, u11_1);
        vfma(ds11, x2, u11_2);
        vfma(ds11, x3, u11_3);
        if (gw) gw[11 * NQV] = ds11;
        vfma(dxp[1], s11, u11_1);
        vfma(dxp[2], s11, u11_2);
        vfma(dxp[3], s11, u11_3);
        const EVec s12 = ss[12 * NQV];  // path 12: l1=1 l2=3 -> L=3
        const EVec sx12_1 = vmul(s12, x1);
        EVec u12_1; vzero(u12_1);
        const EVec sx12_2 = vmul(s12, x2);
        EVec u12_2; vzero(u12_2);
        const EVec sx12_3 = vmul(s12, x3);
        EVec u12_3; vzero(u12_3);
        const EVec d12_24 = dms[24 * NQV];
        vfma(u12_1, a10.z, d12_24);
        { const float t = vdot(sx12_1, d12_24);
          dyl[10] = fmaf(0.353553385f, t, dyl[10]);
        }
        const EVec d12_25 = dms[25 * NQV];
        const float4 a11 = *reinterpret_cast<const float4*>(As + 44);
        vfma(u12_1, a11.y, d12_25);
        { const float t = vdot(sx12_1, d12_25);
          dyl[9] = fmaf(-0.353553385f, t, dyl[9]);
          dyl[11] = fmaf(0.456435472f, t, dyl[11]);
        }
        const EVec d12_26 = dms[26 * NQV];
        const float4 a12 = *reinterpret_cast<const float4*>(As + 48);
        vfma(u12_1, a12.x, d12_26);
        { const float t = vdot(sx12_1, d12_26);
          dyl[10] = fmaf(-0.456435472f, t, dyl[10]);
        }
        const EVec d12_27 = dms[27 * NQV];
        vfma(u12_1, a12.w, d12_27);
        { const float t = vdot(sx12_1, d12_27);
          dyl[13] = fmaf(-0.707106769f, t, dyl[13]);
        }
        const EVec d12_28 = dms[28 * NQV];
        const float4 a13 = *reinterpret_cast<const float4*>(As + 52);
        vfma(u12_1, a13.y, d12_28);
        { const float t = vdot(sx12_1, d12_28);
          dyl[12] = fmaf(0.707106769f, t, dyl[12]);
          dyl[14] = fmaf(-0.456435472f, t, dyl[14]);
        }
        const EVec d12_29 = dms[29 * NQV];
        const float4 a14 = *reinterpret_cast<const float4*>(As + 56);
        vfma(u12_1, a14.x, d12_29);
        { const float t = vdot(sx12_1, d12_29);
          dyl[13] = fmaf(0.456435472f, t, dyl[13]);
          dyl[15] = fmaf(-0.353553385f, t, dyl[15]);
        }
        const EVec d12_30 = dms[30 * NQV];
        vfma(u12_1, a14.w, d12_30);
        { const float t = vdot(sx12_1, d12_30);
          dyl[14] = fmaf(0.353553385f, t, dyl[14]);
        }
        vfma(u12_2, a10.w, d12_24);
        { const float t = vdot(sx12_2, d12_24);
          dyl[15] = fmaf(0.866025388f, t, dyl[15]);
        }
        vfma(u12_2, a11.z, d12_25);
        { const float t = vdot(sx12_2, d12_25);
          dyl[14] = fmaf(0.577350259f, t, dyl[14]);
        }
        vfma(u12_2, a12.y, d12_26);
        { const float t = vdot(sx12_2, d12_26);
          dyl[13] = fmaf(0.288675129f, t, dyl[13]);
        }
        vfma(u12_3, a13.x, d12_27);
        { const float t = vdot(sx12_3, d12_27);
          dyl[11] = fmaf(0.707106769f, t, dyl[11]);
        }
        vfma(u12_2, a13.z, d12_28);
        { const float t = vdot(sx12_2, d12_28);
          dyl[11] = fmaf(-0.288675129f, t, dyl[11]);
        }
        vfma(u12_2, a14.y, d12_29);
        { const float t = vdot(sx12_2, d12_29);
          dyl[10] = fmaf(-0.577350259f, t, dyl[10]);
        }
        const float4 a15 = *reinterpret_cast<const float4*>(As + 60);
        vfma(u12_2, a15.x, d12_30);
        { const float t = vdot(sx12_2, d12_30);
          dyl[9] = fmaf(-0.866025388f, t, dyl[9]);
        }
        vfma(u12_3, a11.x, d12_24);
        { const float t = vdot(sx12_3, d12_24);
          dyl[14] = fmaf(-0.353553385f, t, dyl[14]);
        }
        vfma(u12_3, a11.w, d12_25);
        { const float t = vdot(sx12_3, d12_25);
          dyl[13] = fmaf(-0.456435472f, t, dyl[13]);
          dyl[15] = fmaf(-0.353553385f, t, dyl[15]);
        }
        vfma(u12_3, a12.z, d12_26);
        { const float t = vdot(sx12_3, d12_26);
          dyl[12] = fmaf(-0.707106769f, t, dyl[12]);
          dyl[14] = fmaf(-0.456435472f, t, dyl[14]);
        }
        vfma(u12_3, a13.w, d12_28);
        { const float t = vdot(sx12_3, d12_28);
          dyl[10] = fmaf(0.456435472f, t, dyl[10]);
        }
        vfma(u12_3, a14.z, d12_29);
        { const float t = vdot(sx12_3, d12_29);
          dyl[9] = fmaf(0.353553385f, t, dyl[9]);
          dyl[11] = fmaf(0.456435472f, t, dyl[11]);
        }
        vfma(u12_3, a15.y, d12_30);
        { const float t = vdot(sx12_3, d12_30);
          dyl[10] = fmaf(0.353553385f, t, dyl[10]);
        }
        EVec ds12 = vmul(x1, u12_1);
        vfma(ds12, x2, u12_2);
        vfma(ds12, x3, u12_3);
        if (gw) gw[12 * NQV] = ds12;
        vfma(dxp[1], s12, u12_1);
        vfma(dxp[2], s12, u12_2);
        vfma(dxp[3], s12, u12_3);
    }
};
}  // namespace
}  // namespace fast

extern const FastKernels kFast_w128_l3_collapsed;
const FastKernels kFast_w128_l3_collapsed = {
    "128|0e+1o|3|0:0:0,1:1:0,0:1:1,1:0:1,1:2:1,1:1:1,0:2:2,1:1:2,1:3:2,1:2:2,0:3:3,1:2:3,1:3:3|collapsed",
    &fast::fwd_scratch_bytes<fast::Sig_w128_l3_collapsed>, &fast::bwd_scratch_bytes<fast::Sig_w128_l3_collapsed>, &fast::launch_fwd<fast::Sig_w128_l3_collapsed>, &fast::launch_bwd<fast::Sig_w128_l3_collapsed>, &fast::launch_tp_fwd<fast::Sig_w128_l3_collapsed>, &fast::launch_tp_bwd<fast::Sig_w128_l3_collapsed>,
    nullptr, nullptr, nullptr, nullptr, 0};
}  // namespace e3j
