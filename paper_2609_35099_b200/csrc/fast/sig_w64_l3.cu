// GENERATED by csrc/gen_fast.py from fast/signatures.json -- do not edit.
// signature: 64|0e+1o|3|0:0:0,1:1:0,0:1:1,1:0:1,1:2:1,1:1:1,0:2:2,1:1:2,1:3:2,1:2:2,0:3:3,1:2:3,1:3:3
// 64x0e+64x1o (x) harmonics l<=3: P=13 D=55 nnz=134 pairs=116
#include "fast_fwd.cuh"
#include "fast_bwd.cuh"
#include "fast_launch.cuh"
#include "fast_bwd1s.cuh"

namespace e3j {
namespace fast {
namespace {
__device__ const PairRec kPair_w64_l3[120] = {
    {0,1}, {1,1}, {2,1}, {3,1}, {4,1}, {5,1}, {6,1}, {7,1}, {8,1}, {9,1}, {10,2}, {12,1}, {13,1}, {14,1}, {15,1}, {16,1}, {17,1}, {18,1}, {19,2}, {21,1}, {22,1}, {23,1}, {24,1}, {25,0}, {25,1}, {26,1}, {27,1}, {28,1}, {29,1}, {30,1}, {31,1}, {32,1}, {33,1}, {34,1}, {35,1}, {36,1}, {37,1}, {38,1}, {39,1}, {40,1}, {41,1}, {42,1}, {43,0}, {43,0}, {43,2}, {45,1}, {46,2}, {48,2}, {50,1}, {51,1}, {52,1}, {53,1}, {54,1}, {55,1}, {56,1}, {57,2}, {59,2}, {61,1}, {62,2}, {64,1}, {65,1}, {66,1}, {67,1}, {68,1}, {69,2}, {71,1}, {72,1}, {73,2}, {75,1}, {76,1}, {77,1}, {78,1}, {79,1}, {80,1}, {81,1}, {82,1}, {83,1}, {84,1}, {85,1}, {86,0}, {86,1}, {87,1}, {88,1}, {89,1}, {90,1}, {91,1}, {92,2}, {94,1}, {95,1}, {96,1}, {97,1}, {98,1}, {99,1}, {100,1}, {101,2}, {103,1}, {104,1}, {105,1}, {106,1}, {107,1}, {108,1}, {109,1}, {110,1}, {111,2}, {113,1}, {114,2}, {116,1}, {117,1}, {118,2}, {120,1}, {121,1}, {122,2}, {124,1}, {125,1}, {126,2}, {128,1}, {129,2}, {131,1}, {132,1}, {133,1}};
__device__ const float kVal_w64_l3[134] = {
    1.0f, 0.577350259f, 0.577350259f, 0.577350259f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 0.316227764f, 0.547722578f, -0.547722578f, -0.547722578f, -0.547722578f, -0.632455528f, -0.547722578f, -0.547722578f, -0.547722578f, 0.316227764f, -0.547722578f, 0.707106769f, -0.707106769f, -0.707106769f, 0.707106769f, 0.707106769f, -0.707106769f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 0.707106769f, 0.707106769f, 0.707106769f, 0.707106769f, -0.408248305f, 0.816496611f, -0.408248305f, 0.707106769f, 0.707106769f, -0.707106769f, 0.707106769f, 0.154303357f, 0.597614288f, -0.487950027f, -0.597614288f, 0.154303357f, 0.377964467f, 0.487950027f, -0.617213428f, -0.487950027f, -0.534522474f, -0.654653668f, -0.534522474f, -0.487950027f, -0.617213428f, 0.377964467f, -0.487950027f, -0.597614288f, -0.154303357f, -0.487950027f, 0.154303357f, -0.597614288f, 0.408248305f, 0.816496611f, -0.408248305f, -0.408248305f, 0.408248305f, -0.707106769f, -0.408248305f, -0.707106769f, 0.707106769f, 0.707106769f, -0.408248305f, -0.408248305f, 0.408248305f, 0.408248305f, -0.816496611f, 0.408248305f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 0.707106769f, 0.707106769f, 0.577350259f, 0.577350259f, 0.577350259f, 0.632455528f, 0.182574183f, 0.730296731f, -0.182574183f, -0.44721359f, 0.774596691f, -0.44721359f, -0.182574183f, 0.730296731f, 0.632455528f, -0.182574183f, -0.577350259f, 0.577350259f, 0.577350259f, -0.707106769f, 0.707106769f, 0.353553385f, 0.866025388f, -0.353553385f, -0.353553385f, 0.456435472f, 0.577350259f, -0.456435472f, -0.353553385f, -0.456435472f, 0.288675129f, -0.707106769f, -0.456435472f, -0.707106769f, 0.707106769f, 0.707106769f, -0.456435472f, -0.288675129f, 0.456435472f, 0.456435472f, -0.353553385f, -0.577350259f, 0.353553385f, 0.456435472f, 0.353553385f, -0.866025388f, 0.353553385f};
__device__ const unsigned char kI2_w64_l3[134] = {
    0, 1, 2, 3, 1, 2, 3, 0, 0, 0, 6, 8, 5, 4, 5, 6, 7, 4, 7, 6, 8, 3, 2, 3, 1, 2, 1, 4, 5, 6, 7, 8, 3, 1, 2, 1, 1, 2, 3, 3, 2, 1, 3, 13, 15, 10, 9, 11, 12, 14, 11, 10, 11, 12, 13, 10, 13, 12, 14, 9, 11, 14, 13, 15, 5, 8, 7, 4, 7, 6, 8, 7, 5, 6, 8, 5, 4, 7, 4, 5, 9, 10, 11, 12, 13, 14, 15, 8, 4, 7, 4, 5, 6, 8, 5, 4, 5, 6, 7, 4, 7, 6, 8, 5, 8, 7, 4, 8, 10, 15, 14, 9, 11, 14, 13, 15, 10, 13, 12, 14, 13, 11, 12, 14, 11, 10, 13, 15, 10, 9, 11, 14, 9, 10};
__device__ const PairRec kBPair_w64_l3[124] = {
    {0,1}, {1,1}, {2,1}, {3,1}, {4,1}, {5,1}, {6,1}, {7,1}, {8,1}, {9,1}, {10,1}, {11,1}, {12,1}, {13,1}, {14,1}, {15,1}, {16,1}, {17,1}, {18,1}, {19,1}, {20,2}, {22,1}, {23,1}, {24,2}, {26,1}, {27,1}, {28,1}, {29,1}, {30,1}, {31,0}, {31,0}, {31,0}, {31,1}, {32,1}, {33,1}, {34,1}, {35,1}, {36,1}, {37,1}, {38,1}, {39,1}, {40,1}, {41,1}, {42,1}, {43,1}, {44,2}, {46,1}, {47,2}, {49,1}, {50,1}, {51,2}, {53,1}, {54,1}, {55,2}, {57,1}, {58,1}, {59,2}, {61,1}, {62,2}, {64,1}, {65,1}, {66,1}, {67,0}, {67,0}, {67,1}, {68,1}, {69,1}, {70,1}, {71,1}, {72,1}, {73,1}, {74,1}, {75,1}, {76,1}, {77,1}, {78,1}, {79,1}, {80,1}, {81,2}, {83,1}, {84,1}, {85,1}, {86,1}, {87,1}, {88,1}, {89,1}, {90,2}, {92,1}, {93,1}, {94,1}, {95,1}, {96,1}, {97,2}, {99,1}, {100,1}, {101,1}, {102,1}, {103,1}, {104,1}, {105,1}, {106,2}, {108,1}, {109,1}, {110,1}, {111,1}, {112,1}, {113,2}, {115,1}, {116,2}, {118,2}, {120,1}, {121,1}, {122,1}, {123,1}, {124,1}, {125,1}, {126,1}, {127,2}, {129,2}, {131,1}, {132,2}, {134,0}, {134,0}, {134,0}};
__device__ const float kBVal_w64_l3[134] = {
    1.0f, 1.0f, 1.0f, 1.0f, 0.707106769f, 0.707106769f, 0.707106769f, 0.707106769f, -0.408248305f, 0.816496611f, -0.408248305f, 0.707106769f, 0.707106769f, -0.707106769f, 0.707106769f, 0.408248305f, 0.816496611f, -0.408248305f, -0.408248305f, 0.408248305f, -0.707106769f, -0.408248305f, -0.707106769f, 0.707106769f, 0.707106769f, -0.408248305f, -0.408248305f, 0.408248305f, 0.408248305f, -0.816496611f, 0.408248305f, 0.577350259f, 0.577350259f, 0.577350259f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 0.353553385f, 0.866025388f, -0.353553385f, -0.353553385f, 0.456435472f, 0.577350259f, -0.456435472f, -0.353553385f, -0.456435472f, 0.288675129f, -0.707106769f, -0.456435472f, -0.707106769f, 0.707106769f, 0.707106769f, -0.456435472f, -0.288675129f, 0.456435472f, 0.456435472f, -0.353553385f, -0.577350259f, 0.353553385f, 0.456435472f, 0.353553385f, -0.866025388f, 0.353553385f, 1.0f, 1.0f, 1.0f, 0.707106769f, -0.707106769f, -0.707106769f, 0.707106769f, 0.707106769f, -0.707106769f, 0.707106769f, 0.707106769f, 0.577350259f, 0.577350259f, 0.577350259f, 0.632455528f, 0.182574183f, 0.730296731f, -0.182574183f, -0.44721359f, 0.774596691f, -0.44721359f, -0.182574183f, 0.730296731f, 0.632455528f, -0.182574183f, -0.577350259f, 0.577350259f, 0.577350259f, -0.707106769f, 0.707106769f, 0.316227764f, 0.547722578f, -0.547722578f, -0.547722578f, -0.547722578f, -0.632455528f, -0.547722578f, -0.547722578f, -0.547722578f, 0.316227764f, -0.547722578f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 0.154303357f, 0.597614288f, -0.487950027f, -0.597614288f, 0.154303357f, 0.377964467f, 0.487950027f, -0.617213428f, -0.487950027f, -0.534522474f, -0.654653668f, -0.534522474f, -0.487950027f, -0.617213428f, 0.377964467f, -0.487950027f, -0.597614288f, -0.154303357f, -0.487950027f, 0.154303357f, -0.597614288f};
__device__ const unsigned char kBI2_w64_l3[134] = {
    0, 1, 2, 3, 3, 1, 2, 1, 1, 2, 3, 3, 2, 1, 3, 5, 8, 7, 4, 7, 6, 8, 7, 5, 6, 8, 5, 4, 7, 4, 5, 1, 2, 3, 9, 10, 11, 12, 13, 14, 15, 10, 15, 14, 9, 11, 14, 13, 15, 10, 13, 12, 14, 13, 11, 12, 14, 11, 10, 13, 15, 10, 9, 11, 14, 9, 10, 0, 0, 0, 3, 2, 3, 1, 2, 1, 8, 4, 7, 4, 5, 6, 8, 5, 4, 5, 6, 7, 4, 7, 6, 8, 5, 8, 7, 4, 8, 6, 8, 5, 4, 5, 6, 7, 4, 7, 6, 8, 4, 5, 6, 7, 8, 13, 15, 10, 9, 11, 12, 14, 11, 10, 11, 12, 13, 10, 13, 12, 14, 9, 11, 14, 13, 15};
__device__ const unsigned char kBRow_w64_l3[60] = {
    0, 2, 3, 4, 19, 20, 21, 22, 23, 29, 30, 31, 32, 33, 33, 1, 34, 35, 36, 37, 38, 39, 40, 48, 49, 50, 51, 52, 53, 54, 5, 6, 7, 11, 12, 13, 41, 42, 43, 44, 45, 46, 47, 47, 47, 8, 9, 10, 14, 15, 16, 17, 18, 24, 25, 26, 27, 28, 28, 28};

struct Sig_w64_l3 {
    static constexpr int NQ = 64, DIN = 4, DSH = 16, P = 13, D = 55;
    static constexpr int NNZ = 134, NPAIR = 116, V = 2;
    static constexpr int FW = 4, FT = 10, FS = 2, FC = 2, F_RMAX = 16, F_APAD = 120, F_NREC = 2, F_NPMAX = 40, F_MAXREG = 255;
    // fused double backward (cotangent of grad_out): tile, stages, CTAs per SM (DFT = 0: not generated)
    static constexpr int DFT = 5, DFS = 2, DFC = 2, DFV = 2;
    using DFVec = float2;
    using Vec = float2;
    __device__ static __forceinline__ PairRec pair_rec(int i) { return kPair_w64_l3[i]; }
    __device__ static __forceinline__ float rec_val(int i) { return kVal_w64_l3[i]; }
    __device__ static __forceinline__ unsigned char rec_i2(int i) { return kI2_w64_l3[i]; }
    static constexpr int f_row0(int g) {
        switch (g) {
            case 0: return 0;
            case 1: return 13;
            case 2: return 24;
            case 3: return 40;
            case 4: return 55;
            default: return 55;
        }
    }
    static constexpr int f_a0(int g) {
        switch (g) {
            case 0: return 0;
            case 1: return 24;
            case 2: return 44;
            case 3: return 80;
            case 4: return 120;
            default: return 120;
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
            const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
            pfma(acc[9], a3.y, sx4_1);
            const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
            pfma(acc[10], a4.x, sx4_1);
            pfma(acc[8], a2.w, sx4_2);
            pfma(acc[9], a3.z, sx4_2);
            pfma(acc[10], a4.y, sx4_2);
            pfma(acc[8], a3.x, sx4_3);
            pfma(acc[9], a3.w, sx4_3);
            pfma(acc[10], a4.z, sx4_3);
            const Vec s5 = ss[5 * NQV];  // path 5: l1=1 l2=1 -> L=1
            const Vec sx5_1 = pmul(s5, x1);
            const Vec sx5_2 = pmul(s5, x2);
            const Vec sx5_3 = pmul(s5, x3);
            pfma(acc[11], a4.w, sx5_2);
            const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
            pfma(acc[12], a5.y, sx5_1);
            pfma(acc[11], a5.x, sx5_3);
            pfma(acc[12], a5.z, sx5_3);
        }
        if constexpr (G == 1) {
            const Vec x0 = xs[0 * NQV];
            const Vec x1 = xs[1 * NQV];
            const Vec x2 = xs[2 * NQV];
            const Vec x3 = xs[3 * NQV];
            const Vec s5 = ss[5 * NQV];  // path 5: l1=1 l2=1 -> L=1
            const Vec sx5_1 = pmul(s5, x1);
            const Vec sx5_2 = pmul(s5, x2);
            const float4 a6 = *reinterpret_cast<const float4*>(As + 24);
            pfma(acc[0], a6.x, sx5_1);
            pfma(acc[0], a6.y, sx5_2);
            const Vec s6 = ss[6 * NQV];  // path 6: l1=0 l2=2 -> L=2
            const Vec sx6_0 = pmul(s6, x0);
            pfma(acc[1], a6.z, sx6_0);
            pfma(acc[2], a6.w, sx6_0);
            const float4 a7 = *reinterpret_cast<const float4*>(As + 28);
            pfma(acc[3], a7.x, sx6_0);
            pfma(acc[4], a7.y, sx6_0);
            pfma(acc[5], a7.z, sx6_0);
            const Vec s7 = ss[7 * NQV];  // path 7: l1=1 l2=1 -> L=2
            const Vec sx7_1 = pmul(s7, x1);
            const Vec sx7_2 = pmul(s7, x2);
            const Vec sx7_3 = pmul(s7, x3);
            pfma(acc[6], a7.w, sx7_1);
            const float4 a8 = *reinterpret_cast<const float4*>(As + 32);
            pfma(acc[7], a8.y, sx7_1);
            pfma(acc[8], a8.w, sx7_1);
            const float4 a9 = *reinterpret_cast<const float4*>(As + 36);
            pfma(acc[9], a9.z, sx7_2);
            const float4 a10 = *reinterpret_cast<const float4*>(As + 40);
            pfma(acc[10], a10.x, sx7_1);
            pfma(acc[6], a8.x, sx7_3);
            pfma(acc[7], a8.z, sx7_2);
            pfma(acc[8], a9.x, sx7_2);
            pfma(acc[9], a9.w, sx7_3);
            pfma(acc[10], a10.y, sx7_3);
            pfma(acc[8], a9.y, sx7_3);
        }
        if constexpr (G == 2) {
            const Vec x0 = xs[0 * NQV];
            const Vec x1 = xs[1 * NQV];
            const Vec x2 = xs[2 * NQV];
            const Vec x3 = xs[3 * NQV];
            const Vec s8 = ss[8 * NQV];  // path 8: l1=1 l2=3 -> L=2
            const Vec sx8_1 = pmul(s8, x1);
            const Vec sx8_2 = pmul(s8, x2);
            const Vec sx8_3 = pmul(s8, x3);
            const float4 a11 = *reinterpret_cast<const float4*>(As + 44);
            pfma(acc[0], a11.x, sx8_1);
            pfma(acc[1], a11.w, sx8_1);
            const float4 a12 = *reinterpret_cast<const float4*>(As + 48);
            pfma(acc[2], a12.z, sx8_1);
            const float4 a13 = *reinterpret_cast<const float4*>(As + 52);
            pfma(acc[3], a13.y, sx8_1);
            const float4 a14 = *reinterpret_cast<const float4*>(As + 56);
            pfma(acc[4], a14.x, sx8_1);
            pfma(acc[0], a11.y, sx8_2);
            pfma(acc[1], a12.x, sx8_2);
            pfma(acc[2], a12.w, sx8_2);
            pfma(acc[3], a13.z, sx8_2);
            pfma(acc[4], a14.y, sx8_2);
            pfma(acc[0], a11.z, sx8_3);
            pfma(acc[1], a12.y, sx8_3);
            pfma(acc[2], a13.x, sx8_3);
            pfma(acc[3], a13.w, sx8_3);
            pfma(acc[4], a14.z, sx8_3);
            const Vec s9 = ss[9 * NQV];  // path 9: l1=1 l2=2 -> L=2
            const Vec sx9_1 = pmul(s9, x1);
            const Vec sx9_2 = pmul(s9, x2);
            const Vec sx9_3 = pmul(s9, x3);
            pfma(acc[5], a14.w, sx9_1);
            const float4 a15 = *reinterpret_cast<const float4*>(As + 60);
            pfma(acc[6], a15.z, sx9_1);
            const float4 a16 = *reinterpret_cast<const float4*>(As + 64);
            pfma(acc[7], a16.y, sx9_1);
            pfma(acc[8], a16.w, sx9_1);
            const float4 a17 = *reinterpret_cast<const float4*>(As + 68);
            pfma(acc[9], a17.z, sx9_1);
            pfma(acc[5], a15.x, sx9_2);
            pfma(acc[6], a15.w, sx9_2);
            pfma(acc[7], a16.z, sx9_3);
            pfma(acc[8], a17.x, sx9_2);
            pfma(acc[9], a17.w, sx9_2);
            pfma(acc[5], a15.y, sx9_3);
            pfma(acc[6], a16.x, sx9_3);
            pfma(acc[8], a17.y, sx9_3);
            const float4 a18 = *reinterpret_cast<const float4*>(As + 72);
            pfma(acc[9], a18.x, sx9_3);
            const Vec s10 = ss[10 * NQV];  // path 10: l1=0 l2=3 -> L=3
            const Vec sx10_0 = pmul(s10, x0);
            pfma(acc[10], a18.y, sx10_0);
            pfma(acc[11], a18.z, sx10_0);
            pfma(acc[12], a18.w, sx10_0);
            const float4 a19 = *reinterpret_cast<const float4*>(As + 76);
            pfma(acc[13], a19.x, sx10_0);
            pfma(acc[14], a19.y, sx10_0);
            pfma(acc[15], a19.z, sx10_0);
        }
        if constexpr (G == 3) {
            const Vec x0 = xs[0 * NQV];
            const Vec x1 = xs[1 * NQV];
            const Vec x2 = xs[2 * NQV];
            const Vec x3 = xs[3 * NQV];
            const Vec s10 = ss[10 * NQV];  // path 10: l1=0 l2=3 -> L=3
            const Vec sx10_0 = pmul(s10, x0);
            const float4 a20 = *reinterpret_cast<const float4*>(As + 80);
            pfma(acc[0], a20.x, sx10_0);
            const Vec s11 = ss[11 * NQV];  // path 11: l1=1 l2=2 -> L=3
            const Vec sx11_1 = pmul(s11, x1);
            const Vec sx11_2 = pmul(s11, x2);
            const Vec sx11_3 = pmul(s11, x3);
            pfma(acc[1], a20.y, sx11_1);
            pfma(acc[2], a20.w, sx11_1);
            const float4 a21 = *reinterpret_cast<const float4*>(As + 84);
            pfma(acc[3], a21.z, sx11_1);
            const float4 a22 = *reinterpret_cast<const float4*>(As + 88);
            pfma(acc[4], a22.y, sx11_1);
            const float4 a23 = *reinterpret_cast<const float4*>(As + 92);
            pfma(acc[5], a23.x, sx11_1);
            pfma(acc[6], a23.w, sx11_1);
            const float4 a24 = *reinterpret_cast<const float4*>(As + 96);
            pfma(acc[7], a24.z, sx11_1);
            pfma(acc[1], a20.z, sx11_3);
            pfma(acc[2], a21.x, sx11_2);
            pfma(acc[3], a21.w, sx11_2);
            pfma(acc[4], a22.z, sx11_2);
            pfma(acc[5], a23.y, sx11_2);
            pfma(acc[6], a24.x, sx11_2);
            pfma(acc[7], a24.w, sx11_3);
            pfma(acc[2], a21.y, sx11_3);
            pfma(acc[3], a22.x, sx11_3);
            pfma(acc[4], a22.w, sx11_3);
            pfma(acc[5], a23.z, sx11_3);
            pfma(acc[6], a24.y, sx11_3);
            const Vec s12 = ss[12 * NQV];  // path 12: l1=1 l2=3 -> L=3
            const Vec sx12_1 = pmul(s12, x1);
            const Vec sx12_2 = pmul(s12, x2);
            const Vec sx12_3 = pmul(s12, x3);
            const float4 a25 = *reinterpret_cast<const float4*>(As + 100);
            pfma(acc[8], a25.x, sx12_1);
            pfma(acc[9], a25.w, sx12_1);
            const float4 a26 = *reinterpret_cast<const float4*>(As + 104);
            pfma(acc[10], a26.z, sx12_1);
            const float4 a27 = *reinterpret_cast<const float4*>(As + 108);
            pfma(acc[11], a27.y, sx12_1);
            pfma(acc[12], a27.w, sx12_1);
            const float4 a28 = *reinterpret_cast<const float4*>(As + 112);
            pfma(acc[13], a28.z, sx12_1);
            const float4 a29 = *reinterpret_cast<const float4*>(As + 116);
            pfma(acc[14], a29.y, sx12_1);
            pfma(acc[8], a25.y, sx12_2);
            pfma(acc[9], a26.x, sx12_2);
            pfma(acc[10], a26.w, sx12_2);
            pfma(acc[11], a27.z, sx12_3);
            pfma(acc[12], a28.x, sx12_2);
            pfma(acc[13], a28.w, sx12_2);
            pfma(acc[14], a29.z, sx12_2);
            pfma(acc[8], a25.z, sx12_3);
            pfma(acc[9], a26.y, sx12_3);
            pfma(acc[10], a27.x, sx12_3);
            pfma(acc[12], a28.y, sx12_3);
            pfma(acc[13], a29.x, sx12_3);
            pfma(acc[14], a29.w, sx12_3);
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
            const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
            const float4 b3 = *reinterpret_cast<const float4*>(Bs + 12);
            pfma(acc[9], a3.y, sxu4_1);
            pfma(acc[9], b3.y, sx4_1);
            const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
            const float4 b4 = *reinterpret_cast<const float4*>(Bs + 16);
            pfma(acc[10], a4.x, sxu4_1);
            pfma(acc[10], b4.x, sx4_1);
            pfma(acc[8], a2.w, sxu4_2);
            pfma(acc[8], b2.w, sx4_2);
            pfma(acc[9], a3.z, sxu4_2);
            pfma(acc[9], b3.z, sx4_2);
            pfma(acc[10], a4.y, sxu4_2);
            pfma(acc[10], b4.y, sx4_2);
            pfma(acc[8], a3.x, sxu4_3);
            pfma(acc[8], b3.x, sx4_3);
            pfma(acc[9], a3.w, sxu4_3);
            pfma(acc[9], b3.w, sx4_3);
            pfma(acc[10], a4.z, sxu4_3);
            pfma(acc[10], b4.z, sx4_3);
            const DFVec s5 = ss[5 * NQV];
            const DFVec us5 = uss[5 * NQV];
            const DFVec sx5_1 = pmul(s5, x1);
            DFVec sxu5_1 = pmul(s5, ux1); pfma(sxu5_1, us5, x1);
            const DFVec sx5_2 = pmul(s5, x2);
            DFVec sxu5_2 = pmul(s5, ux2); pfma(sxu5_2, us5, x2);
            const DFVec sx5_3 = pmul(s5, x3);
            DFVec sxu5_3 = pmul(s5, ux3); pfma(sxu5_3, us5, x3);
            pfma(acc[11], a4.w, sxu5_2);
            pfma(acc[11], b4.w, sx5_2);
            const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
            const float4 b5 = *reinterpret_cast<const float4*>(Bs + 20);
            pfma(acc[12], a5.y, sxu5_1);
            pfma(acc[12], b5.y, sx5_1);
            pfma(acc[11], a5.x, sxu5_3);
            pfma(acc[11], b5.x, sx5_3);
            pfma(acc[12], a5.z, sxu5_3);
            pfma(acc[12], b5.z, sx5_3);
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
            const DFVec s5 = ss[5 * NQV];
            const DFVec us5 = uss[5 * NQV];
            const DFVec sx5_1 = pmul(s5, x1);
            DFVec sxu5_1 = pmul(s5, ux1); pfma(sxu5_1, us5, x1);
            const DFVec sx5_2 = pmul(s5, x2);
            DFVec sxu5_2 = pmul(s5, ux2); pfma(sxu5_2, us5, x2);
            const float4 a6 = *reinterpret_cast<const float4*>(As + 24);
            const float4 b6 = *reinterpret_cast<const float4*>(Bs + 24);
            pfma(acc[0], a6.x, sxu5_1);
            pfma(acc[0], b6.x, sx5_1);
            pfma(acc[0], a6.y, sxu5_2);
            pfma(acc[0], b6.y, sx5_2);
            const DFVec s6 = ss[6 * NQV];
            const DFVec us6 = uss[6 * NQV];
            const DFVec sx6_0 = pmul(s6, x0);
            DFVec sxu6_0 = pmul(s6, ux0); pfma(sxu6_0, us6, x0);
            pfma(acc[1], a6.z, sxu6_0);
            pfma(acc[1], b6.z, sx6_0);
            pfma(acc[2], a6.w, sxu6_0);
            pfma(acc[2], b6.w, sx6_0);
            const float4 a7 = *reinterpret_cast<const float4*>(As + 28);
            const float4 b7 = *reinterpret_cast<const float4*>(Bs + 28);
            pfma(acc[3], a7.x, sxu6_0);
            pfma(acc[3], b7.x, sx6_0);
            pfma(acc[4], a7.y, sxu6_0);
            pfma(acc[4], b7.y, sx6_0);
            pfma(acc[5], a7.z, sxu6_0);
            pfma(acc[5], b7.z, sx6_0);
            const DFVec s7 = ss[7 * NQV];
            const DFVec us7 = uss[7 * NQV];
            const DFVec sx7_1 = pmul(s7, x1);
            DFVec sxu7_1 = pmul(s7, ux1); pfma(sxu7_1, us7, x1);
            const DFVec sx7_2 = pmul(s7, x2);
            DFVec sxu7_2 = pmul(s7, ux2); pfma(sxu7_2, us7, x2);
            const DFVec sx7_3 = pmul(s7, x3);
            DFVec sxu7_3 = pmul(s7, ux3); pfma(sxu7_3, us7, x3);
            pfma(acc[6], a7.w, sxu7_1);
            pfma(acc[6], b7.w, sx7_1);
            const float4 a8 = *reinterpret_cast<const float4*>(As + 32);
            const float4 b8 = *reinterpret_cast<const float4*>(Bs + 32);
            pfma(acc[7], a8.y, sxu7_1);
            pfma(acc[7], b8.y, sx7_1);
            pfma(acc[8], a8.w, sxu7_1);
            pfma(acc[8], b8.w, sx7_1);
            const float4 a9 = *reinterpret_cast<const float4*>(As + 36);
            const float4 b9 = *reinterpret_cast<const float4*>(Bs + 36);
            pfma(acc[9], a9.z, sxu7_2);
            pfma(acc[9], b9.z, sx7_2);
            const float4 a10 = *reinterpret_cast<const float4*>(As + 40);
            const float4 b10 = *reinterpret_cast<const float4*>(Bs + 40);
            pfma(acc[10], a10.x, sxu7_1);
            pfma(acc[10], b10.x, sx7_1);
            pfma(acc[6], a8.x, sxu7_3);
            pfma(acc[6], b8.x, sx7_3);
            pfma(acc[7], a8.z, sxu7_2);
            pfma(acc[7], b8.z, sx7_2);
            pfma(acc[8], a9.x, sxu7_2);
            pfma(acc[8], b9.x, sx7_2);
            pfma(acc[9], a9.w, sxu7_3);
            pfma(acc[9], b9.w, sx7_3);
            pfma(acc[10], a10.y, sxu7_3);
            pfma(acc[10], b10.y, sx7_3);
            pfma(acc[8], a9.y, sxu7_3);
            pfma(acc[8], b9.y, sx7_3);
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
            const DFVec s8 = ss[8 * NQV];
            const DFVec us8 = uss[8 * NQV];
            const DFVec sx8_1 = pmul(s8, x1);
            DFVec sxu8_1 = pmul(s8, ux1); pfma(sxu8_1, us8, x1);
            const DFVec sx8_2 = pmul(s8, x2);
            DFVec sxu8_2 = pmul(s8, ux2); pfma(sxu8_2, us8, x2);
            const DFVec sx8_3 = pmul(s8, x3);
            DFVec sxu8_3 = pmul(s8, ux3); pfma(sxu8_3, us8, x3);
            const float4 a11 = *reinterpret_cast<const float4*>(As + 44);
            const float4 b11 = *reinterpret_cast<const float4*>(Bs + 44);
            pfma(acc[0], a11.x, sxu8_1);
            pfma(acc[0], b11.x, sx8_1);
            pfma(acc[1], a11.w, sxu8_1);
            pfma(acc[1], b11.w, sx8_1);
            const float4 a12 = *reinterpret_cast<const float4*>(As + 48);
            const float4 b12 = *reinterpret_cast<const float4*>(Bs + 48);
            pfma(acc[2], a12.z, sxu8_1);
            pfma(acc[2], b12.z, sx8_1);
            const float4 a13 = *reinterpret_cast<const float4*>(As + 52);
            const float4 b13 = *reinterpret_cast<const float4*>(Bs + 52);
            pfma(acc[3], a13.y, sxu8_1);
            pfma(acc[3], b13.y, sx8_1);
            const float4 a14 = *reinterpret_cast<const float4*>(As + 56);
            const float4 b14 = *reinterpret_cast<const float4*>(Bs + 56);
            pfma(acc[4], a14.x, sxu8_1);
            pfma(acc[4], b14.x, sx8_1);
            pfma(acc[0], a11.y, sxu8_2);
            pfma(acc[0], b11.y, sx8_2);
            pfma(acc[1], a12.x, sxu8_2);
            pfma(acc[1], b12.x, sx8_2);
            pfma(acc[2], a12.w, sxu8_2);
            pfma(acc[2], b12.w, sx8_2);
            pfma(acc[3], a13.z, sxu8_2);
            pfma(acc[3], b13.z, sx8_2);
            pfma(acc[4], a14.y, sxu8_2);
            pfma(acc[4], b14.y, sx8_2);
            pfma(acc[0], a11.z, sxu8_3);
            pfma(acc[0], b11.z, sx8_3);
            pfma(acc[1], a12.y, sxu8_3);
            pfma(acc[1], b12.y, sx8_3);
            pfma(acc[2], a13.x, sxu8_3);
            pfma(acc[2], b13.x, sx8_3);
            pfma(acc[3], a13.w, sxu8_3);
            pfma(acc[3], b13.w, sx8_3);
            pfma(acc[4], a14.z, sxu8_3);
            pfma(acc[4], b14.z, sx8_3);
            const DFVec s9 = ss[9 * NQV];
            const DFVec us9 = uss[9 * NQV];
            const DFVec sx9_1 = pmul(s9, x1);
            DFVec sxu9_1 = pmul(s9, ux1); pfma(sxu9_1, us9, x1);
            const DFVec sx9_2 = pmul(s9, x2);
            DFVec sxu9_2 = pmul(s9, ux2); pfma(sxu9_2, us9, x2);
            const DFVec sx9_3 = pmul(s9, x3);
            DFVec sxu9_3 = pmul(s9, ux3); pfma(sxu9_3, us9, x3);
            pfma(acc[5], a14.w, sxu9_1);
            pfma(acc[5], b14.w, sx9_1);
            const float4 a15 = *reinterpret_cast<const float4*>(As + 60);
            const float4 b15 = *reinterpret_cast<const float4*>(Bs + 60);
            pfma(acc[6], a15.z, sxu9_1);
            pfma(acc[6], b15.z, sx9_1);
            const float4 a16 = *reinterpret_cast<const float4*>(As + 64);
            const float4 b16 = *reinterpret_cast<const float4*>(Bs + 64);
            pfma(acc[7], a16.y, sxu9_1);
            pfma(acc[7], b16.y, sx9_1);
            pfma(acc[8], a16.w, sxu9_1);
            pfma(acc[8], b16.w, sx9_1);
            const float4 a17 = *reinterpret_cast<const float4*>(As + 68);
            const float4 b17 = *reinterpret_cast<const float4*>(Bs + 68);
            pfma(acc[9], a17.z, sxu9_1);
            pfma(acc[9], b17.z, sx9_1);
            pfma(acc[5], a15.x, sxu9_2);
            pfma(acc[5], b15.x, sx9_2);
            pfma(acc[6], a15.w, sxu9_2);
            pfma(acc[6], b15.w, sx9_2);
            pfma(acc[7], a16.z, sxu9_3);
            pfma(acc[7], b16.z, sx9_3);
            pfma(acc[8], a17.x, sxu9_2);
            pfma(acc[8], b17.x, sx9_2);
            pfma(acc[9], a17.w, sxu9_2);
            pfma(acc[9], b17.w, sx9_2);
            pfma(acc[5], a15.y, sxu9_3);
            pfma(acc[5], b15.y, sx9_3);
            pfma(acc[6], a16.x, sxu9_3);
            pfma(acc[6], b16.x, sx9_3);
            pfma(acc[8], a17.y, sxu9_3);
            pfma(acc[8], b17.y, sx9_3);
            const float4 a18 = *reinterpret_cast<const float4*>(As + 72);
            const float4 b18 = *reinterpret_cast<const float4*>(Bs + 72);
            pfma(acc[9], a18.x, sxu9_3);
            pfma(acc[9], b18.x, sx9_3);
            const DFVec s10 = ss[10 * NQV];
            const DFVec us10 = uss[10 * NQV];
            const DFVec sx10_0 = pmul(s10, x0);
            DFVec sxu10_0 = pmul(s10, ux0); pfma(sxu10_0, us10, x0);
            pfma(acc[10], a18.y, sxu10_0);
            pfma(acc[10], b18.y, sx10_0);
            pfma(acc[11], a18.z, sxu10_0);
            pfma(acc[11], b18.z, sx10_0);
            pfma(acc[12], a18.w, sxu10_0);
            pfma(acc[12], b18.w, sx10_0);
            const float4 a19 = *reinterpret_cast<const float4*>(As + 76);
            const float4 b19 = *reinterpret_cast<const float4*>(Bs + 76);
            pfma(acc[13], a19.x, sxu10_0);
            pfma(acc[13], b19.x, sx10_0);
            pfma(acc[14], a19.y, sxu10_0);
            pfma(acc[14], b19.y, sx10_0);
            pfma(acc[15], a19.z, sxu10_0);
            pfma(acc[15], b19.z, sx10_0);
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
            const DFVec s10 = ss[10 * NQV];
            const DFVec us10 = uss[10 * NQV];
            const DFVec sx10_0 = pmul(s10, x0);
            DFVec sxu10_0 = pmul(s10, ux0); pfma(sxu10_0, us10, x0);
            const float4 a20 = *reinterpret_cast<const float4*>(As + 80);
            const float4 b20 = *reinterpret_cast<const float4*>(Bs + 80);
            pfma(acc[0], a20.x, sxu10_0);
            pfma(acc[0], b20.x, sx10_0);
            const DFVec s11 = ss[11 * NQV];
            const DFVec us11 = uss[11 * NQV];
            const DFVec sx11_1 = pmul(s11, x1);
            DFVec sxu11_1 = pmul(s11, ux1); pfma(sxu11_1, us11, x1);
            const DFVec sx11_2 = pmul(s11, x2);
            DFVec sxu11_2 = pmul(s11, ux2); pfma(sxu11_2, us11, x2);
            const DFVec sx11_3 = pmul(s11, x3);
            DFVec sxu11_3 = pmul(s11, ux3); pfma(sxu11_3, us11, x3);
            pfma(acc[1], a20.y, sxu11_1);
            pfma(acc[1], b20.y, sx11_1);
            pfma(acc[2], a20.w, sxu11_1);
            pfma(acc[2], b20.w, sx11_1);
            const float4 a21 = *reinterpret_cast<const float4*>(As + 84);
            const float4 b21 = *reinterpret_cast<const float4*>(Bs + 84);
            pfma(acc[3], a21.z, sxu11_1);
            pfma(acc[3], b21.z, sx11_1);
            const float4 a22 = *reinterpret_cast<const float4*>(As + 88);
            const float4 b22 = *reinterpret_cast<const float4*>(Bs + 88);
            pfma(acc[4], a22.y, sxu11_1);
            pfma(acc[4], b22.y, sx11_1);
            const float4 a23 = *reinterpret_cast<const float4*>(As + 92);
            const float4 b23 = *reinterpret_cast<const float4*>(Bs + 92);
            pfma(acc[5], a23.x, sxu11_1);
            pfma(acc[5], b23.x, sx11_1);
            pfma(acc[6], a23.w, sxu11_1);
            pfma(acc[6], b23.w, sx11_1);
            const float4 a24 = *reinterpret_cast<const float4*>(As + 96);
            const float4 b24 = *reinterpret_cast<const float4*>(Bs + 96);
            pfma(acc[7], a24.z, sxu11_1);
            pfma(acc[7], b24.z, sx11_1);
            pfma(acc[1], a20.z, sxu11_3);
            pfma(acc[1], b20.z, sx11_3);
            pfma(acc[2], a21.x, sxu11_2);
            pfma(acc[2], b21.x, sx11_2);
            pfma(acc[3], a21.w, sxu11_2);
            pfma(acc[3], b21.w, sx11_2);
            pfma(acc[4], a22.z, sxu11_2);
            pfma(acc[4], b22.z, sx11_2);
            pfma(acc[5], a23.y, sxu11_2);
            pfma(acc[5], b23.y, sx11_2);
            pfma(acc[6], a24.x, sxu11_2);
            pfma(acc[6], b24.x, sx11_2);
            pfma(acc[7], a24.w, sxu11_3);
            pfma(acc[7], b24.w, sx11_3);
            pfma(acc[2], a21.y, sxu11_3);
            pfma(acc[2], b21.y, sx11_3);
            pfma(acc[3], a22.x, sxu11_3);
            pfma(acc[3], b22.x, sx11_3);
            pfma(acc[4], a22.w, sxu11_3);
            pfma(acc[4], b22.w, sx11_3);
            pfma(acc[5], a23.z, sxu11_3);
            pfma(acc[5], b23.z, sx11_3);
            pfma(acc[6], a24.y, sxu11_3);
            pfma(acc[6], b24.y, sx11_3);
            const DFVec s12 = ss[12 * NQV];
            const DFVec us12 = uss[12 * NQV];
            const DFVec sx12_1 = pmul(s12, x1);
            DFVec sxu12_1 = pmul(s12, ux1); pfma(sxu12_1, us12, x1);
            const DFVec sx12_2 = pmul(s12, x2);
            DFVec sxu12_2 = pmul(s12, ux2); pfma(sxu12_2, us12, x2);
            const DFVec sx12_3 = pmul(s12, x3);
            DFVec sxu12_3 = pmul(s12, ux3); pfma(sxu12_3, us12, x3);
            const float4 a25 = *reinterpret_cast<const float4*>(As + 100);
            const float4 b25 = *reinterpret_cast<const float4*>(Bs + 100);
            pfma(acc[8], a25.x, sxu12_1);
            pfma(acc[8], b25.x, sx12_1);
            pfma(acc[9], a25.w, sxu12_1);
            pfma(acc[9], b25.w, sx12_1);
            const float4 a26 = *reinterpret_cast<const float4*>(As + 104);
            const float4 b26 = *reinterpret_cast<const float4*>(Bs + 104);
            pfma(acc[10], a26.z, sxu12_1);
            pfma(acc[10], b26.z, sx12_1);
            const float4 a27 = *reinterpret_cast<const float4*>(As + 108);
            const float4 b27 = *reinterpret_cast<const float4*>(Bs + 108);
            pfma(acc[11], a27.y, sxu12_1);
            pfma(acc[11], b27.y, sx12_1);
            pfma(acc[12], a27.w, sxu12_1);
            pfma(acc[12], b27.w, sx12_1);
            const float4 a28 = *reinterpret_cast<const float4*>(As + 112);
            const float4 b28 = *reinterpret_cast<const float4*>(Bs + 112);
            pfma(acc[13], a28.z, sxu12_1);
            pfma(acc[13], b28.z, sx12_1);
            const float4 a29 = *reinterpret_cast<const float4*>(As + 116);
            const float4 b29 = *reinterpret_cast<const float4*>(Bs + 116);
            pfma(acc[14], a29.y, sxu12_1);
            pfma(acc[14], b29.y, sx12_1);
            pfma(acc[8], a25.y, sxu12_2);
            pfma(acc[8], b25.y, sx12_2);
            pfma(acc[9], a26.x, sxu12_2);
            pfma(acc[9], b26.x, sx12_2);
            pfma(acc[10], a26.w, sxu12_2);
            pfma(acc[10], b26.w, sx12_2);
            pfma(acc[11], a27.z, sxu12_3);
            pfma(acc[11], b27.z, sx12_3);
            pfma(acc[12], a28.x, sxu12_2);
            pfma(acc[12], b28.x, sx12_2);
            pfma(acc[13], a28.w, sxu12_2);
            pfma(acc[13], b28.w, sx12_2);
            pfma(acc[14], a29.z, sxu12_2);
            pfma(acc[14], b29.z, sx12_2);
            pfma(acc[8], a25.z, sxu12_3);
            pfma(acc[8], b25.z, sx12_3);
            pfma(acc[9], a26.y, sxu12_3);
            pfma(acc[9], b26.y, sx12_3);
            pfma(acc[10], a27.x, sxu12_3);
            pfma(acc[10], b27.x, sx12_3);
            pfma(acc[12], a28.y, sxu12_3);
            pfma(acc[12], b28.y, sx12_3);
            pfma(acc[13], a29.x, sxu12_3);
            pfma(acc[13], b29.x, sx12_3);
            pfma(acc[14], a29.w, sxu12_3);
            pfma(acc[14], b29.w, sx12_3);
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
            dst[9 * stride] = acc[9];
            dst[10 * stride] = acc[10];
            dst[11 * stride] = acc[11];
            dst[12 * stride] = acc[12];
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
            dst[10 * stride] = acc[10];
            dst[11 * stride] = acc[11];
            dst[12 * stride] = acc[12];
            dst[13 * stride] = acc[13];
            dst[14 * stride] = acc[14];
            dst[15 * stride] = acc[15];
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
            dst[11 * stride] = acc[11];
            dst[12 * stride] = acc[12];
            dst[13 * stride] = acc[13];
            dst[14 * stride] = acc[14];
        }
    }
    // ---- backward: path groups [[0, 2, 7, 9], [1, 10, 12], [3, 5, 11], [4, 6, 8]]
    static constexpr int BV = 2;  // channels per lane in the backward
    using BVec = float2;
    static constexpr int BW = 4, BT = 8, BS = 2, BC = 2, B_RMAX = 15, B_APAD = 124, B_NREC = 2;
    // edge-wise backward (one warp per edge, grad_out rows read from shared memory): edges per tile (0 = not generated), ring stages
    static constexpr int ET = 15, ES = 2, EV = 2, EXG = 1;   // EXG: sender rows not staged
    static constexpr int ST = 10;   // columns of the scheduled backward
    // the same for the standalone tensor product: rows per ring slot (0 = not generated), ring slots
    static constexpr int ETR = 0, ESR = 3;
    // fused double backward (edge outputs): edges per tile (0 = not generated), ring stages
    static constexpr int DT = 8, DS = 2, DV = 2;
    using DVec = float2;
    using EVec = float2;
    __device__ static __forceinline__ PairRec b_pair_rec(int i) { return kBPair_w64_l3[i]; }
    __device__ static __forceinline__ float b_rec_val(int i) { return kBVal_w64_l3[i]; }
    __device__ static __forceinline__ unsigned char b_rec_i2(int i) { return kBI2_w64_l3[i]; }
    // output rows of path group g: b_nrow(g) of them, the r-th is b_row(g, r)
    __device__ static __forceinline__ int b_row(int g, int r) { return kBRow_w64_l3[g * B_RMAX + r]; }
    static constexpr int b_nrow(int g) {
        switch (g) {
            case 0: return 14;
            case 1: return 15;
            case 2: return 13;
            case 3: return 13;
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
            const BVec s5 = ss[5 * NQV];  // path 5: l1=1 l2=1 -> L=1
            const BVec sx5_1 = vmul(s5, x1);
            BVec u5_1; vzero(u5_1);
            const BVec sx5_2 = vmul(s5, x2);
            BVec u5_2; vzero(u5_2);
            const BVec sx5_3 = vmul(s5, x3);
            BVec u5_3; vzero(u5_3);
            vfma(u5_2, a16.w, dm[3]);
            { const float t = vdot(sx5_2, dm[3]);
              dyl[3] = 0.707106769f * t;
            }
            const float4 a17 = *reinterpret_cast<const float4*>(As + 68);
            vfma(u5_1, a17.y, dm[4]);
            { const float t = vdot(sx5_1, dm[4]);
              dyl[3] = fmaf(-0.707106769f, t, dyl[3]);
            }
            vfma(u5_1, a17.w, dm[5]);
            { const float t = vdot(sx5_1, dm[5]);
              dyl[2] = 0.707106769f * t;
            }
            vfma(u5_3, a17.x, dm[3]);
            { const float t = vdot(sx5_3, dm[3]);
              dyl[2] = fmaf(-0.707106769f, t, dyl[2]);
            }
            vfma(u5_3, a17.z, dm[4]);
            { const float t = vdot(sx5_3, dm[4]);
              dyl[1] = 0.707106769f * t;
            }
            const float4 a18 = *reinterpret_cast<const float4*>(As + 72);
            vfma(u5_2, a18.x, dm[5]);
            { const float t = vdot(sx5_2, dm[5]);
              dyl[1] = fmaf(-0.707106769f, t, dyl[1]);
            }
            BVec ds5 = vmul(x1, u5_1);
            vfma(ds5, x2, u5_2);
            vfma(ds5, x3, u5_3);
            if (gw) gw[5 * NQV] = ds5;
            vfma(dxp[1], s5, u5_1);
            vfma(dxp[2], s5, u5_2);
            vfma(dxp[3], s5, u5_3);
            const BVec s11 = ss[11 * NQV];  // path 11: l1=1 l2=2 -> L=3
            const BVec sx11_1 = vmul(s11, x1);
            BVec u11_1; vzero(u11_1);
            const BVec sx11_2 = vmul(s11, x2);
            BVec u11_2; vzero(u11_2);
            const BVec sx11_3 = vmul(s11, x3);
            BVec u11_3; vzero(u11_3);
            vfma(u11_1, a18.y, dm[6]);
            { const float t = vdot(sx11_1, dm[6]);
              dyl[8] = 0.707106769f * t;
            }
            vfma(u11_1, a18.w, dm[7]);
            { const float t = vdot(sx11_1, dm[7]);
              dyl[7] = 0.577350259f * t;
            }
            const float4 a19 = *reinterpret_cast<const float4*>(As + 76);
            vfma(u11_1, a19.z, dm[8]);
            { const float t = vdot(sx11_1, dm[8]);
              dyl[6] = 0.632455528f * t;
              dyl[8] = fmaf(0.182574183f, t, dyl[8]);
            }
            const float4 a20 = *reinterpret_cast<const float4*>(As + 80);
            vfma(u11_1, a20.y, dm[9]);
            { const float t = vdot(sx11_1, dm[9]);
              dyl[5] = -0.44721359f * t;
            }
            const float4 a21 = *reinterpret_cast<const float4*>(As + 84);
            vfma(u11_1, a21.x, dm[10]);
            { const float t = vdot(sx11_1, dm[10]);
              dyl[4] = -0.182574183f * t;
            }
            vfma(u11_1, a21.w, dm[11]);
            { const float t = vdot(sx11_1, dm[11]);
              dyl[5] = fmaf(-0.577350259f, t, dyl[5]);
            }
            const float4 a22 = *reinterpret_cast<const float4*>(As + 88);
            vfma(u11_1, a22.z, dm[12]);
            { const float t = vdot(sx11_1, dm[12]);
              dyl[4] = fmaf(-0.707106769f, t, dyl[4]);
            }
            vfma(u11_3, a18.z, dm[6]);
            { const float t = vdot(sx11_3, dm[6]);
              dyl[4] = fmaf(0.707106769f, t, dyl[4]);
            }
            vfma(u11_2, a19.x, dm[7]);
            { const float t = vdot(sx11_2, dm[7]);
              dyl[4] = fmaf(0.577350259f, t, dyl[4]);
            }
            vfma(u11_2, a19.w, dm[8]);
            { const float t = vdot(sx11_2, dm[8]);
              dyl[5] = fmaf(0.730296731f, t, dyl[5]);
            }
            vfma(u11_2, a20.z, dm[9]);
            { const float t = vdot(sx11_2, dm[9]);
              dyl[6] = fmaf(0.774596691f, t, dyl[6]);
            }
            vfma(u11_2, a21.y, dm[10]);
            { const float t = vdot(sx11_2, dm[10]);
              dyl[7] = fmaf(0.730296731f, t, dyl[7]);
            }
            vfma(u11_2, a22.x, dm[11]);
            { const float t = vdot(sx11_2, dm[11]);
              dyl[8] = fmaf(0.577350259f, t, dyl[8]);
            }
            vfma(u11_3, a22.w, dm[12]);
            { const float t = vdot(sx11_3, dm[12]);
              dyl[8] = fmaf(0.707106769f, t, dyl[8]);
            }
            vfma(u11_3, a19.y, dm[7]);
            { const float t = vdot(sx11_3, dm[7]);
              dyl[5] = fmaf(0.577350259f, t, dyl[5]);
            }
            vfma(u11_3, a20.x, dm[8]);
            { const float t = vdot(sx11_3, dm[8]);
              dyl[4] = fmaf(-0.182574183f, t, dyl[4]);
            }
            vfma(u11_3, a20.w, dm[9]);
            { const float t = vdot(sx11_3, dm[9]);
              dyl[7] = fmaf(-0.44721359f, t, dyl[7]);
            }
            vfma(u11_3, a21.z, dm[10]);
            { const float t = vdot(sx11_3, dm[10]);
              dyl[6] = fmaf(0.632455528f, t, dyl[6]);
              dyl[8] = fmaf(-0.182574183f, t, dyl[8]);
            }
            vfma(u11_3, a22.y, dm[11]);
            { const float t = vdot(sx11_3, dm[11]);
              dyl[7] = fmaf(0.577350259f, t, dyl[7]);
            }
            BVec ds11 = vmul(x1, u11_1);
            vfma(ds11, x2, u11_2);
            vfma(ds11, x3, u11_3);
            if (gw) gw[11 * NQV] = ds11;
            vfma(dxp[1], s11, u11_1);
            vfma(dxp[2], s11, u11_2);
            vfma(dxp[3], s11, u11_3);
            vzero(dxp[0]);
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
            const BVec s4 = ss[4 * NQV];  // path 4: l1=1 l2=2 -> L=1
            const BVec sx4_1 = vmul(s4, x1);
            BVec u4_1; vzero(u4_1);
            const BVec sx4_2 = vmul(s4, x2);
            BVec u4_2; vzero(u4_2);
            const BVec sx4_3 = vmul(s4, x3);
            BVec u4_3; vzero(u4_3);
            const float4 a23 = *reinterpret_cast<const float4*>(As + 92);
            vfma(u4_1, a23.x, dm[0]);
            { const float t = vdot(sx4_1, dm[0]);
              dyl[6] = 0.316227764f * t;
              dyl[8] = 0.547722578f * t;
            }
            vfma(u4_1, a23.w, dm[1]);
            { const float t = vdot(sx4_1, dm[1]);
              dyl[5] = -0.547722578f * t;
            }
            const float4 a24 = *reinterpret_cast<const float4*>(As + 96);
            vfma(u4_1, a24.z, dm[2]);
            { const float t = vdot(sx4_1, dm[2]);
              dyl[4] = -0.547722578f * t;
            }
            vfma(u4_2, a23.y, dm[0]);
            { const float t = vdot(sx4_2, dm[0]);
              dyl[5] = fmaf(-0.547722578f, t, dyl[5]);
            }
            vfma(u4_2, a24.x, dm[1]);
            { const float t = vdot(sx4_2, dm[1]);
              dyl[6] = fmaf(-0.632455528f, t, dyl[6]);
            }
            vfma(u4_2, a24.w, dm[2]);
            { const float t = vdot(sx4_2, dm[2]);
              dyl[7] = -0.547722578f * t;
            }
            vfma(u4_3, a23.z, dm[0]);
            { const float t = vdot(sx4_3, dm[0]);
              dyl[4] = fmaf(-0.547722578f, t, dyl[4]);
            }
            vfma(u4_3, a24.y, dm[1]);
            { const float t = vdot(sx4_3, dm[1]);
              dyl[7] = fmaf(-0.547722578f, t, dyl[7]);
            }
            const float4 a25 = *reinterpret_cast<const float4*>(As + 100);
            vfma(u4_3, a25.x, dm[2]);
            { const float t = vdot(sx4_3, dm[2]);
              dyl[6] = fmaf(0.316227764f, t, dyl[6]);
              dyl[8] = fmaf(-0.547722578f, t, dyl[8]);
            }
            BVec ds4 = vmul(x1, u4_1);
            vfma(ds4, x2, u4_2);
            vfma(ds4, x3, u4_3);
            if (gw) gw[4 * NQV] = ds4;
            dxp[1] = vmul(s4, u4_1);
            dxp[2] = vmul(s4, u4_2);
            dxp[3] = vmul(s4, u4_3);
            const BVec s6 = ss[6 * NQV];  // path 6: l1=0 l2=2 -> L=2
            const BVec sx6_0 = vmul(s6, x0);
            BVec u6_0; vzero(u6_0);
            vfma(u6_0, a25.y, dm[3]);
            { const float t = vdot(sx6_0, dm[3]);
              dyl[4] = fmaf(1.0f, t, dyl[4]);
            }
            vfma(u6_0, a25.z, dm[4]);
            { const float t = vdot(sx6_0, dm[4]);
              dyl[5] = fmaf(1.0f, t, dyl[5]);
            }
            vfma(u6_0, a25.w, dm[5]);
            { const float t = vdot(sx6_0, dm[5]);
              dyl[6] = fmaf(1.0f, t, dyl[6]);
            }
            const float4 a26 = *reinterpret_cast<const float4*>(As + 104);
            vfma(u6_0, a26.x, dm[6]);
            { const float t = vdot(sx6_0, dm[6]);
              dyl[7] = fmaf(1.0f, t, dyl[7]);
            }
            vfma(u6_0, a26.y, dm[7]);
            { const float t = vdot(sx6_0, dm[7]);
              dyl[8] = fmaf(1.0f, t, dyl[8]);
            }
            BVec ds6 = vmul(x0, u6_0);
            if (gw) gw[6 * NQV] = ds6;
            dxp[0] = vmul(s6, u6_0);
            const BVec s8 = ss[8 * NQV];  // path 8: l1=1 l2=3 -> L=2
            const BVec sx8_1 = vmul(s8, x1);
            BVec u8_1; vzero(u8_1);
            const BVec sx8_2 = vmul(s8, x2);
            BVec u8_2; vzero(u8_2);
            const BVec sx8_3 = vmul(s8, x3);
            BVec u8_3; vzero(u8_3);
            vfma(u8_1, a26.z, dm[8]);
            { const float t = vdot(sx8_1, dm[8]);
              dyl[13] = 0.154303357f * t;
              dyl[15] = 0.597614288f * t;
            }
            const float4 a27 = *reinterpret_cast<const float4*>(As + 108);
            vfma(u8_1, a27.y, dm[9]);
            { const float t = vdot(sx8_1, dm[9]);
              dyl[12] = 0.377964467f * t;
              dyl[14] = 0.487950027f * t;
            }
            const float4 a28 = *reinterpret_cast<const float4*>(As + 112);
            vfma(u8_1, a28.x, dm[10]);
            { const float t = vdot(sx8_1, dm[10]);
              dyl[11] = -0.534522474f * t;
            }
            vfma(u8_1, a28.w, dm[11]);
            { const float t = vdot(sx8_1, dm[11]);
              dyl[10] = -0.487950027f * t;
            }
            const float4 a29 = *reinterpret_cast<const float4*>(As + 116);
            vfma(u8_1, a29.z, dm[12]);
            { const float t = vdot(sx8_1, dm[12]);
              dyl[9] = -0.597614288f * t;
              dyl[11] = fmaf(-0.154303357f, t, dyl[11]);
            }
            vfma(u8_2, a26.w, dm[8]);
            { const float t = vdot(sx8_2, dm[8]);
              dyl[10] = fmaf(-0.487950027f, t, dyl[10]);
            }
            vfma(u8_2, a27.z, dm[9]);
            { const float t = vdot(sx8_2, dm[9]);
              dyl[11] = fmaf(-0.617213428f, t, dyl[11]);
            }
            vfma(u8_2, a28.y, dm[10]);
            { const float t = vdot(sx8_2, dm[10]);
              dyl[12] = fmaf(-0.654653668f, t, dyl[12]);
            }
            vfma(u8_2, a29.x, dm[11]);
            { const float t = vdot(sx8_2, dm[11]);
              dyl[13] = fmaf(-0.617213428f, t, dyl[13]);
            }
            vfma(u8_2, a29.w, dm[12]);
            { const float t = vdot(sx8_2, dm[12]);
              dyl[14] = fmaf(-0.487950027f, t, dyl[14]);
            }
            vfma(u8_3, a27.x, dm[8]);
            { const float t = vdot(sx8_3, dm[8]);
              dyl[9] = fmaf(-0.597614288f, t, dyl[9]);
              dyl[11] = fmaf(0.154303357f, t, dyl[11]);
            }
            vfma(u8_3, a27.w, dm[9]);
            { const float t = vdot(sx8_3, dm[9]);
              dyl[10] = fmaf(-0.487950027f, t, dyl[10]);
            }
            vfma(u8_3, a28.z, dm[10]);
            { const float t = vdot(sx8_3, dm[10]);
              dyl[13] = fmaf(-0.534522474f, t, dyl[13]);
            }
            vfma(u8_3, a29.y, dm[11]);
            { const float t = vdot(sx8_3, dm[11]);
              dyl[12] = fmaf(0.377964467f, t, dyl[12]);
              dyl[14] = fmaf(-0.487950027f, t, dyl[14]);
            }
            const float4 a30 = *reinterpret_cast<const float4*>(As + 120);
            vfma(u8_3, a30.x, dm[12]);
            { const float t = vdot(sx8_3, dm[12]);
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
            dyl[0] = 0.f;
            dyl[1] = 0.f;
            dyl[2] = 0.f;
            dyl[3] = 0.f;
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
        float2 dyv[16];
        const EVec s0 = ss[0 * NQV];  // path 0: l1=0 l2=0 -> L=0
        const EVec sx0_0 = pmul(s0, x0);
        EVec u0_0; vzero(u0_0);
        const EVec d0_0 = dms[0 * NQV];
        const float4 a0 = *reinterpret_cast<const float4*>(As + 0);
        pfma(u0_0, a0.x, d0_0);
        { const float2 t = pmul(sx0_0, d0_0);
          vzero(dyv[0]);
          pfma(dyv[0], 1.0f, t);
        }
        EVec ds0 = pmul(x0, u0_0);
        if (gw) gw[0 * NQV] = ds0;
        dxp[0] = pmul(s0, u0_0);
        const EVec s1 = ss[1 * NQV];  // path 1: l1=1 l2=1 -> L=0
        const EVec sx1_1 = pmul(s1, x1);
        EVec u1_1; vzero(u1_1);
        const EVec sx1_2 = pmul(s1, x2);
        EVec u1_2; vzero(u1_2);
        const EVec sx1_3 = pmul(s1, x3);
        EVec u1_3; vzero(u1_3);
        const EVec d1_1 = dms[1 * NQV];
        const float4 a8 = *reinterpret_cast<const float4*>(As + 32);
        pfma(u1_1, a8.x, d1_1);
        { const float2 t = pmul(sx1_1, d1_1);
          vzero(dyv[1]);
          pfma(dyv[1], 0.577350259f, t);
        }
        pfma(u1_2, a8.y, d1_1);
        { const float2 t = pmul(sx1_2, d1_1);
          vzero(dyv[2]);
          pfma(dyv[2], 0.577350259f, t);
        }
        pfma(u1_3, a8.z, d1_1);
        { const float2 t = pmul(sx1_3, d1_1);
          vzero(dyv[3]);
          pfma(dyv[3], 0.577350259f, t);
        }
        EVec ds1 = pmul(x1, u1_1);
        pfma(ds1, x2, u1_2);
        pfma(ds1, x3, u1_3);
        if (gw) gw[1 * NQV] = ds1;
        dxp[1] = pmul(s1, u1_1);
        dxp[2] = pmul(s1, u1_2);
        dxp[3] = pmul(s1, u1_3);
        const EVec s2 = ss[2 * NQV];  // path 2: l1=0 l2=1 -> L=1
        const EVec sx2_0 = pmul(s2, x0);
        EVec u2_0; vzero(u2_0);
        const EVec d2_2 = dms[2 * NQV];
        pfma(u2_0, a0.y, d2_2);
        { const float2 t = pmul(sx2_0, d2_2);
          pfma(dyv[1], 1.0f, t);
        }
        const EVec d2_3 = dms[3 * NQV];
        pfma(u2_0, a0.z, d2_3);
        { const float2 t = pmul(sx2_0, d2_3);
          pfma(dyv[2], 1.0f, t);
        }
        const EVec d2_4 = dms[4 * NQV];
        pfma(u2_0, a0.w, d2_4);
        { const float2 t = pmul(sx2_0, d2_4);
          pfma(dyv[3], 1.0f, t);
        }
        EVec ds2 = pmul(x0, u2_0);
        if (gw) gw[2 * NQV] = ds2;
        pfma(dxp[0], s2, u2_0);
        const EVec s3 = ss[3 * NQV];  // path 3: l1=1 l2=0 -> L=1
        const EVec sx3_1 = pmul(s3, x1);
        EVec u3_1; vzero(u3_1);
        const EVec sx3_2 = pmul(s3, x2);
        EVec u3_2; vzero(u3_2);
        const EVec sx3_3 = pmul(s3, x3);
        EVec u3_3; vzero(u3_3);
        const EVec d3_5 = dms[5 * NQV];
        const float4 a16 = *reinterpret_cast<const float4*>(As + 64);
        pfma(u3_1, a16.x, d3_5);
        { const float2 t = pmul(sx3_1, d3_5);
          pfma(dyv[0], 1.0f, t);
        }
        const EVec d3_6 = dms[6 * NQV];
        pfma(u3_2, a16.y, d3_6);
        { const float2 t = pmul(sx3_2, d3_6);
          pfma(dyv[0], 1.0f, t);
        }
        const EVec d3_7 = dms[7 * NQV];
        pfma(u3_3, a16.z, d3_7);
        { const float2 t = pmul(sx3_3, d3_7);
          pfma(dyv[0], 1.0f, t);
        }
        EVec ds3 = pmul(x1, u3_1);
        pfma(ds3, x2, u3_2);
        pfma(ds3, x3, u3_3);
        if (gw) gw[3 * NQV] = ds3;
        pfma(dxp[1], s3, u3_1);
        pfma(dxp[2], s3, u3_2);
        pfma(dxp[3], s3, u3_3);
        const EVec s4 = ss[4 * NQV];  // path 4: l1=1 l2=2 -> L=1
        const EVec sx4_1 = pmul(s4, x1);
        EVec u4_1; vzero(u4_1);
        const EVec sx4_2 = pmul(s4, x2);
        EVec u4_2; vzero(u4_2);
        const EVec sx4_3 = pmul(s4, x3);
        EVec u4_3; vzero(u4_3);
        const EVec d4_8 = dms[8 * NQV];
        const float4 a23 = *reinterpret_cast<const float4*>(As + 92);
        pfma(u4_1, a23.x, d4_8);
        { const float2 t = pmul(sx4_1, d4_8);
          vzero(dyv[6]);
          pfma(dyv[6], 0.316227764f, t);
          vzero(dyv[8]);
          pfma(dyv[8], 0.547722578f, t);
        }
        const EVec d4_9 = dms[9 * NQV];
        pfma(u4_1, a23.w, d4_9);
        { const float2 t = pmul(sx4_1, d4_9);
          vzero(dyv[5]);
          pfma(dyv[5], -0.547722578f, t);
        }
        const EVec d4_10 = dms[10 * NQV];
        const float4 a24 = *reinterpret_cast<const float4*>(As + 96);
        pfma(u4_1, a24.z, d4_10);
        { const float2 t = pmul(sx4_1, d4_10);
          vzero(dyv[4]);
          pfma(dyv[4], -0.547722578f, t);
        }
        pfma(u4_2, a23.y, d4_8);
        { const float2 t = pmul(sx4_2, d4_8);
          pfma(dyv[5], -0.547722578f, t);
        }
        pfma(u4_2, a24.x, d4_9);
        { const float2 t = pmul(sx4_2, d4_9);
          pfma(dyv[6], -0.632455528f, t);
        }
        pfma(u4_2, a24.w, d4_10);
        { const float2 t = pmul(sx4_2, d4_10);
          vzero(dyv[7]);
          pfma(dyv[7], -0.547722578f, t);
        }
        pfma(u4_3, a23.z, d4_8);
        { const float2 t = pmul(sx4_3, d4_8);
          pfma(dyv[4], -0.547722578f, t);
        }
        pfma(u4_3, a24.y, d4_9);
        { const float2 t = pmul(sx4_3, d4_9);
          pfma(dyv[7], -0.547722578f, t);
        }
        const float4 a25 = *reinterpret_cast<const float4*>(As + 100);
        pfma(u4_3, a25.x, d4_10);
        { const float2 t = pmul(sx4_3, d4_10);
          pfma(dyv[6], 0.316227764f, t);
          pfma(dyv[8], -0.547722578f, t);
        }
        EVec ds4 = pmul(x1, u4_1);
        pfma(ds4, x2, u4_2);
        pfma(ds4, x3, u4_3);
        if (gw) gw[4 * NQV] = ds4;
        pfma(dxp[1], s4, u4_1);
        pfma(dxp[2], s4, u4_2);
        pfma(dxp[3], s4, u4_3);
        const EVec s5 = ss[5 * NQV];  // path 5: l1=1 l2=1 -> L=1
        const EVec sx5_1 = pmul(s5, x1);
        EVec u5_1; vzero(u5_1);
        const EVec sx5_2 = pmul(s5, x2);
        EVec u5_2; vzero(u5_2);
        const EVec sx5_3 = pmul(s5, x3);
        EVec u5_3; vzero(u5_3);
        const EVec d5_11 = dms[11 * NQV];
        pfma(u5_2, a16.w, d5_11);
        { const float2 t = pmul(sx5_2, d5_11);
          pfma(dyv[3], 0.707106769f, t);
        }
        const EVec d5_12 = dms[12 * NQV];
        const float4 a17 = *reinterpret_cast<const float4*>(As + 68);
        pfma(u5_1, a17.y, d5_12);
        { const float2 t = pmul(sx5_1, d5_12);
          pfma(dyv[3], -0.707106769f, t);
        }
        const EVec d5_13 = dms[13 * NQV];
        pfma(u5_1, a17.w, d5_13);
        { const float2 t = pmul(sx5_1, d5_13);
          pfma(dyv[2], 0.707106769f, t);
        }
        pfma(u5_3, a17.x, d5_11);
        { const float2 t = pmul(sx5_3, d5_11);
          pfma(dyv[2], -0.707106769f, t);
        }
        pfma(u5_3, a17.z, d5_12);
        { const float2 t = pmul(sx5_3, d5_12);
          pfma(dyv[1], 0.707106769f, t);
        }
        const float4 a18 = *reinterpret_cast<const float4*>(As + 72);
        pfma(u5_2, a18.x, d5_13);
        { const float2 t = pmul(sx5_2, d5_13);
          pfma(dyv[1], -0.707106769f, t);
        }
        EVec ds5 = pmul(x1, u5_1);
        pfma(ds5, x2, u5_2);
        pfma(ds5, x3, u5_3);
        if (gw) gw[5 * NQV] = ds5;
        pfma(dxp[1], s5, u5_1);
        pfma(dxp[2], s5, u5_2);
        pfma(dxp[3], s5, u5_3);
        const EVec s6 = ss[6 * NQV];  // path 6: l1=0 l2=2 -> L=2
        const EVec sx6_0 = pmul(s6, x0);
        EVec u6_0; vzero(u6_0);
        const EVec d6_14 = dms[14 * NQV];
        pfma(u6_0, a25.y, d6_14);
        { const float2 t = pmul(sx6_0, d6_14);
          pfma(dyv[4], 1.0f, t);
        }
        const EVec d6_15 = dms[15 * NQV];
        pfma(u6_0, a25.z, d6_15);
        { const float2 t = pmul(sx6_0, d6_15);
          pfma(dyv[5], 1.0f, t);
        }
        const EVec d6_16 = dms[16 * NQV];
        pfma(u6_0, a25.w, d6_16);
        { const float2 t = pmul(sx6_0, d6_16);
          pfma(dyv[6], 1.0f, t);
        }
        const EVec d6_17 = dms[17 * NQV];
        const float4 a26 = *reinterpret_cast<const float4*>(As + 104);
        pfma(u6_0, a26.x, d6_17);
        { const float2 t = pmul(sx6_0, d6_17);
          pfma(dyv[7], 1.0f, t);
        }
        const EVec d6_18 = dms[18 * NQV];
        pfma(u6_0, a26.y, d6_18);
        { const float2 t = pmul(sx6_0, d6_18);
          pfma(dyv[8], 1.0f, t);
        }
        EVec ds6 = pmul(x0, u6_0);
        if (gw) gw[6 * NQV] = ds6;
        pfma(dxp[0], s6, u6_0);
        const EVec s7 = ss[7 * NQV];  // path 7: l1=1 l2=1 -> L=2
        const EVec sx7_1 = pmul(s7, x1);
        EVec u7_1; vzero(u7_1);
        const EVec sx7_2 = pmul(s7, x2);
        EVec u7_2; vzero(u7_2);
        const EVec sx7_3 = pmul(s7, x3);
        EVec u7_3; vzero(u7_3);
        const EVec d7_19 = dms[19 * NQV];
        const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
        pfma(u7_1, a1.x, d7_19);
        { const float2 t = pmul(sx7_1, d7_19);
          pfma(dyv[3], 0.707106769f, t);
        }
        const EVec d7_20 = dms[20 * NQV];
        pfma(u7_1, a1.z, d7_20);
        { const float2 t = pmul(sx7_1, d7_20);
          pfma(dyv[2], 0.707106769f, t);
        }
        const EVec d7_21 = dms[21 * NQV];
        const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
        pfma(u7_1, a2.x, d7_21);
        { const float2 t = pmul(sx7_1, d7_21);
          pfma(dyv[1], -0.408248305f, t);
        }
        const EVec d7_22 = dms[22 * NQV];
        pfma(u7_2, a2.w, d7_22);
        { const float2 t = pmul(sx7_2, d7_22);
          pfma(dyv[3], 0.707106769f, t);
        }
        const EVec d7_23 = dms[23 * NQV];
        const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
        pfma(u7_1, a3.y, d7_23);
        { const float2 t = pmul(sx7_1, d7_23);
          pfma(dyv[1], -0.707106769f, t);
        }
        pfma(u7_3, a1.y, d7_19);
        { const float2 t = pmul(sx7_3, d7_19);
          pfma(dyv[1], 0.707106769f, t);
        }
        pfma(u7_2, a1.w, d7_20);
        { const float2 t = pmul(sx7_2, d7_20);
          pfma(dyv[1], 0.707106769f, t);
        }
        pfma(u7_2, a2.y, d7_21);
        { const float2 t = pmul(sx7_2, d7_21);
          pfma(dyv[2], 0.816496611f, t);
        }
        pfma(u7_3, a3.x, d7_22);
        { const float2 t = pmul(sx7_3, d7_22);
          pfma(dyv[2], 0.707106769f, t);
        }
        pfma(u7_3, a3.z, d7_23);
        { const float2 t = pmul(sx7_3, d7_23);
          pfma(dyv[3], 0.707106769f, t);
        }
        pfma(u7_3, a2.z, d7_21);
        { const float2 t = pmul(sx7_3, d7_21);
          pfma(dyv[3], -0.408248305f, t);
        }
        EVec ds7 = pmul(x1, u7_1);
        pfma(ds7, x2, u7_2);
        pfma(ds7, x3, u7_3);
        if (gw) gw[7 * NQV] = ds7;
        pfma(dxp[1], s7, u7_1);
        pfma(dxp[2], s7, u7_2);
        pfma(dxp[3], s7, u7_3);
        const EVec s8 = ss[8 * NQV];  // path 8: l1=1 l2=3 -> L=2
        const EVec sx8_1 = pmul(s8, x1);
        EVec u8_1; vzero(u8_1);
        const EVec sx8_2 = pmul(s8, x2);
        EVec u8_2; vzero(u8_2);
        const EVec sx8_3 = pmul(s8, x3);
        EVec u8_3; vzero(u8_3);
        const EVec d8_24 = dms[24 * NQV];
        pfma(u8_1, a26.z, d8_24);
        { const float2 t = pmul(sx8_1, d8_24);
          vzero(dyv[13]);
          pfma(dyv[13], 0.154303357f, t);
          vzero(dyv[15]);
          pfma(dyv[15], 0.597614288f, t);
        }
        const EVec d8_25 = dms[25 * NQV];
        const float4 a27 = *reinterpret_cast<const float4*>(As + 108);
        pfma(u8_1, a27.y, d8_25);
        { const float2 t = pmul(sx8_1, d8_25);
          vzero(dyv[12]);
          pfma(dyv[12], 0.377964467f, t);
          vzero(dyv[14]);
          pfma(dyv[14], 0.487950027f, t);
        }
        const EVec d8_26 = dms[26 * NQV];
        const float4 a28 = *reinterpret_cast<const float4*>(As + 112);
        pfma(u8_1, a28.x, d8_26);
        { const float2 t = pmul(sx8_1, d8_26);
          vzero(dyv[11]);
          pfma(dyv[11], -0.534522474f, t);
        }
        const EVec d8_27 = dms[27 * NQV];
        pfma(u8_1, a28.w, d8_27);
        { const float2 t = pmul(sx8_1, d8_27);
          vzero(dyv[10]);
          pfma(dyv[10], -0.487950027f, t);
        }
        const EVec d8_28 = dms[28 * NQV];
        const float4 a29 = *reinterpret_cast<const float4*>(As + 116);
        pfma(u8_1, a29.z, d8_28);
        { const float2 t = pmul(sx8_1, d8_28);
          vzero(dyv[9]);
          pfma(dyv[9], -0.597614288f, t);
          pfma(dyv[11], -0.154303357f, t);
        }
        pfma(u8_2, a26.w, d8_24);
        { const float2 t = pmul(sx8_2, d8_24);
          pfma(dyv[10], -0.487950027f, t);
        }
        pfma(u8_2, a27.z, d8_25);
        { const float2 t = pmul(sx8_2, d8_25);
          pfma(dyv[11], -0.617213428f, t);
        }
        pfma(u8_2, a28.y, d8_26);
        { const float2 t = pmul(sx8_2, d8_26);
          pfma(dyv[12], -0.654653668f, t);
        }
        pfma(u8_2, a29.x, d8_27);
        { const float2 t = pmul(sx8_2, d8_27);
          pfma(dyv[13], -0.617213428f, t);
        }
        pfma(u8_2, a29.w, d8_28);
        { const float2 t = pmul(sx8_2, d8_28);
          pfma(dyv[14], -0.487950027f, t);
        }
        pfma(u8_3, a27.x, d8_24);
        { const float2 t = pmul(sx8_3, d8_24);
          pfma(dyv[9], -0.597614288f, t);
          pfma(dyv[11], 0.154303357f, t);
        }
        pfma(u8_3, a27.w, d8_25);
        { const float2 t = pmul(sx8_3, d8_25);
          pfma(dyv[10], -0.487950027f, t);
        }
        pfma(u8_3, a28.z, d8_26);
        { const float2 t = pmul(sx8_3, d8_26);
          pfma(dyv[13], -0.534522474f, t);
        }
        pfma(u8_3, a29.y, d8_27);
        { const float2 t = pmul(sx8_3, d8_27);
          pfma(dyv[12], 0.377964467f, t);
          pfma(dyv[14], -0.487950027f, t);
        }
        const float4 a30 = *reinterpret_cast<const float4*>(As + 120);
        pfma(u8_3, a30.x, d8_28);
        { const float2 t = pmul(sx8_3, d8_28);
          pfma(dyv[13], 0.154303357f, t);
          pfma(dyv[15], -0.597614288f, t);
        }
        EVec ds8 = pmul(x1, u8_1);
        pfma(ds8, x2, u8_2);
        pfma(ds8, x3, u8_3);
        if (gw) gw[8 * NQV] = ds8;
        pfma(dxp[1], s8, u8_1);
        pfma(dxp[2], s8, u8_2);
        pfma(dxp[3], s8, u8_3);
        const EVec s9 = ss[9 * NQV];  // path 9: l1=1 l2=2 -> L=2
        const EVec sx9_1 = pmul(s9, x1);
        EVec u9_1; vzero(u9_1);
        const EVec sx9_2 = pmul(s9, x2);
        EVec u9_2; vzero(u9_2);
        const EVec sx9_3 = pmul(s9, x3);
        EVec u9_3; vzero(u9_3);
        const EVec d9_29 = dms[29 * NQV];
        pfma(u9_1, a3.w, d9_29);
        { const float2 t = pmul(sx9_1, d9_29);
          pfma(dyv[5], 0.408248305f, t);
        }
        const EVec d9_30 = dms[30 * NQV];
        const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
        pfma(u9_1, a4.z, d9_30);
        { const float2 t = pmul(sx9_1, d9_30);
          pfma(dyv[4], -0.408248305f, t);
        }
        const EVec d9_31 = dms[31 * NQV];
        const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
        pfma(u9_1, a5.y, d9_31);
        { const float2 t = pmul(sx9_1, d9_31);
          pfma(dyv[7], -0.707106769f, t);
        }
        const EVec d9_32 = dms[32 * NQV];
        pfma(u9_1, a5.w, d9_32);
        { const float2 t = pmul(sx9_1, d9_32);
          pfma(dyv[6], 0.707106769f, t);
          pfma(dyv[8], -0.408248305f, t);
        }
        const EVec d9_33 = dms[33 * NQV];
        const float4 a6 = *reinterpret_cast<const float4*>(As + 24);
        pfma(u9_1, a6.z, d9_33);
        { const float2 t = pmul(sx9_1, d9_33);
          pfma(dyv[7], 0.408248305f, t);
        }
        pfma(u9_2, a4.x, d9_29);
        { const float2 t = pmul(sx9_2, d9_29);
          pfma(dyv[8], 0.816496611f, t);
        }
        pfma(u9_2, a4.w, d9_30);
        { const float2 t = pmul(sx9_2, d9_30);
          pfma(dyv[7], 0.408248305f, t);
        }
        pfma(u9_3, a5.z, d9_31);
        { const float2 t = pmul(sx9_3, d9_31);
          pfma(dyv[5], 0.707106769f, t);
        }
        pfma(u9_2, a6.x, d9_32);
        { const float2 t = pmul(sx9_2, d9_32);
          pfma(dyv[5], -0.408248305f, t);
        }
        pfma(u9_2, a6.w, d9_33);
        { const float2 t = pmul(sx9_2, d9_33);
          pfma(dyv[4], -0.816496611f, t);
        }
        pfma(u9_3, a4.y, d9_29);
        { const float2 t = pmul(sx9_3, d9_29);
          pfma(dyv[7], -0.408248305f, t);
        }
        pfma(u9_3, a5.x, d9_30);
        { const float2 t = pmul(sx9_3, d9_30);
          pfma(dyv[6], -0.707106769f, t);
          pfma(dyv[8], -0.408248305f, t);
        }
        pfma(u9_3, a6.y, d9_32);
        { const float2 t = pmul(sx9_3, d9_32);
          pfma(dyv[4], 0.408248305f, t);
        }
        const float4 a7 = *reinterpret_cast<const float4*>(As + 28);
        pfma(u9_3, a7.x, d9_33);
        { const float2 t = pmul(sx9_3, d9_33);
          pfma(dyv[5], 0.408248305f, t);
        }
        EVec ds9 = pmul(x1, u9_1);
        pfma(ds9, x2, u9_2);
        pfma(ds9, x3, u9_3);
        if (gw) gw[9 * NQV] = ds9;
        pfma(dxp[1], s9, u9_1);
        pfma(dxp[2], s9, u9_2);
        pfma(dxp[3], s9, u9_3);
        const EVec s10 = ss[10 * NQV];  // path 10: l1=0 l2=3 -> L=3
        const EVec sx10_0 = pmul(s10, x0);
        EVec u10_0; vzero(u10_0);
        const EVec d10_34 = dms[34 * NQV];
        pfma(u10_0, a8.w, d10_34);
        { const float2 t = pmul(sx10_0, d10_34);
          pfma(dyv[9], 1.0f, t);
        }
        const EVec d10_35 = dms[35 * NQV];
        const float4 a9 = *reinterpret_cast<const float4*>(As + 36);
        pfma(u10_0, a9.x, d10_35);
        { const float2 t = pmul(sx10_0, d10_35);
          pfma(dyv[10], 1.0f, t);
        }
        const EVec d10_36 = dms[36 * NQV];
        pfma(u10_0, a9.y, d10_36);
        { const float2 t = pmul(sx10_0, d10_36);
          pfma(dyv[11], 1.0f, t);
        }
        const EVec d10_37 = dms[37 * NQV];
        pfma(u10_0, a9.z, d10_37);
        { const float2 t = pmul(sx10_0, d10_37);
          pfma(dyv[12], 1.0f, t);
        }
        const EVec d10_38 = dms[38 * NQV];
        pfma(u10_0, a9.w, d10_38);
        { const float2 t = pmul(sx10_0, d10_38);
          pfma(dyv[13], 1.0f, t);
        }
        const EVec d10_39 = dms[39 * NQV];
        const float4 a10 = *reinterpret_cast<const float4*>(As + 40);
        pfma(u10_0, a10.x, d10_39);
        { const float2 t = pmul(sx10_0, d10_39);
          pfma(dyv[14], 1.0f, t);
        }
        const EVec d10_40 = dms[40 * NQV];
        pfma(u10_0, a10.y, d10_40);
        { const float2 t = pmul(sx10_0, d10_40);
          pfma(dyv[15], 1.0f, t);
        }
        EVec ds10 = pmul(x0, u10_0);
        if (gw) gw[10 * NQV] = ds10;
        pfma(dxp[0], s10, u10_0);
        const EVec s11 = ss[11 * NQV];  // path 11: l1=1 l2=2 -> L=3
        const EVec sx11_1 = pmul(s11, x1);
        EVec u11_1; vzero(u11_1);
        const EVec sx11_2 = pmul(s11, x2);
        EVec u11_2; vzero(u11_2);
        const EVec sx11_3 = pmul(s11, x3);
        EVec u11_3; vzero(u11_3);
        const EVec d11_41 = dms[41 * NQV];
        pfma(u11_1, a18.y, d11_41);
        { const float2 t = pmul(sx11_1, d11_41);
          pfma(dyv[8], 0.707106769f, t);
        }
        const EVec d11_42 = dms[42 * NQV];
        pfma(u11_1, a18.w, d11_42);
        { const float2 t = pmul(sx11_1, d11_42);
          pfma(dyv[7], 0.577350259f, t);
        }
        const EVec d11_43 = dms[43 * NQV];
        const float4 a19 = *reinterpret_cast<const float4*>(As + 76);
        pfma(u11_1, a19.z, d11_43);
        { const float2 t = pmul(sx11_1, d11_43);
          pfma(dyv[6], 0.632455528f, t);
          pfma(dyv[8], 0.182574183f, t);
        }
        const EVec d11_44 = dms[44 * NQV];
        const float4 a20 = *reinterpret_cast<const float4*>(As + 80);
        pfma(u11_1, a20.y, d11_44);
        { const float2 t = pmul(sx11_1, d11_44);
          pfma(dyv[5], -0.44721359f, t);
        }
        const EVec d11_45 = dms[45 * NQV];
        const float4 a21 = *reinterpret_cast<const float4*>(As + 84);
        pfma(u11_1, a21.x, d11_45);
        { const float2 t = pmul(sx11_1, d11_45);
          pfma(dyv[4], -0.182574183f, t);
        }
        const EVec d11_46 = dms[46 * NQV];
        pfma(u11_1, a21.w, d11_46);
        { const float2 t = pmul(sx11_1, d11_46);
          pfma(dyv[5], -0.577350259f, t);
        }
        const EVec d11_47 = dms[47 * NQV];
        const float4 a22 = *reinterpret_cast<const float4*>(As + 88);
        pfma(u11_1, a22.z, d11_47);
        { const float2 t = pmul(sx11_1, d11_47);
          pfma(dyv[4], -0.707106769f, t);
        }
        pfma(u11_3, a18.z, d11_41);
        { const float2 t = pmul(sx11_3, d11_41);
          pfma(dyv[4], 0.707106769f, t);
        }
        pfma(u11_2, a19.x, d11_42);
        { const float2 t = pmul(sx11_2, d11_42);
          pfma(dyv[4], 0.577350259f, t);
        }
        pfma(u11_2, a19.w, d11_43);
        { const float2 t = pmul(sx11_2, d11_43);
          pfma(dyv[5], 0.730296731f, t);
        }
        pfma(u11_2, a20.z, d11_44);
        { const float2 t = pmul(sx11_2, d11_44);
          pfma(dyv[6], 0.774596691f, t);
        }
        pfma(u11_2, a21.y, d11_45);
        { const float2 t = pmul(sx11_2, d11_45);
          pfma(dyv[7], 0.730296731f, t);
        }
        pfma(u11_2, a22.x, d11_46);
        { const float2 t = pmul(sx11_2, d11_46);
          pfma(dyv[8], 0.577350259f, t);
        }
        pfma(u11_3, a22.w, d11_47);
        { const float2 t = pmul(sx11_3, d11_47);
          pfma(dyv[8], 0.707106769f, t);
        }
        pfma(u11_3, a19.y, d11_42);
        { const float2 t = pmul(sx11_3, d11_42);
          pfma(dyv[5], 0.577350259f, t);
        }
        pfma(u11_3, a20.x, d11_43);
        { const float2 t = pmul(sx11_3, d11_43);
          pfma(dyv[4], -0.182574183f, t);
        }
        pfma(u11_3, a20.w, d11_44);
        { const float2 t = pmul(sx11_3, d11_44);
          pfma(dyv[7], -0.44721359f, t);
        }
        pfma(u11_3, a21.z, d11_45);
        { const float2 t = pmul(sx11_3, d11_45);
          pfma(dyv[6], 0.632455528f, t);
          pfma(dyv[8], -0.182574183f, t);
        }
        pfma(u11_3, a22.y, d11_46);
        { const float2 t = pmul(sx11_3, d11_46);
          pfma(dyv[7], 0.577350259f, t);
        }
        EVec ds11 = pmul(x1, u11_1);
        pfma(ds11, x2, u11_2);
        pfma(ds11, x3, u11_3);
        if (gw) gw[11 * NQV] = ds11;
        pfma(dxp[1], s11, u11_1);
        pfma(dxp[2], s11, u11_2);
        pfma(dxp[3], s11, u11_3);
        const EVec s12 = ss[12 * NQV];  // path 12: l1=1 l2=3 -> L=3
        const EVec sx12_1 = pmul(s12, x1);
        EVec u12_1; vzero(u12_1);
        const EVec sx12_2 = pmul(s12, x2);
        EVec u12_2; vzero(u12_2);
        const EVec sx12_3 = pmul(s12, x3);
        EVec u12_3; vzero(u12_3);
        const EVec d12_48 = dms[48 * NQV];
        pfma(u12_1, a10.z, d12_48);
        { const float2 t = pmul(sx12_1, d12_48);
          pfma(dyv[10], 0.353553385f, t);
        }
        const EVec d12_49 = dms[49 * NQV];
        const float4 a11 = *reinterpret_cast<const float4*>(As + 44);
        pfma(u12_1, a11.y, d12_49);
        { const float2 t = pmul(sx12_1, d12_49);
          pfma(dyv[9], -0.353553385f, t);
          pfma(dyv[11], 0.456435472f, t);
        }
        const EVec d12_50 = dms[50 * NQV];
        const float4 a12 = *reinterpret_cast<const float4*>(As + 48);
        pfma(u12_1, a12.x, d12_50);
        { const float2 t = pmul(sx12_1, d12_50);
          pfma(dyv[10], -0.456435472f, t);
        }
        const EVec d12_51 = dms[51 * NQV];
        pfma(u12_1, a12.w, d12_51);
        { const float2 t = pmul(sx12_1, d12_51);
          pfma(dyv[13], -0.707106769f, t);
        }
        const EVec d12_52 = dms[52 * NQV];
        const float4 a13 = *reinterpret_cast<const float4*>(As + 52);
        pfma(u12_1, a13.y, d12_52);
        { const float2 t = pmul(sx12_1, d12_52);
          pfma(dyv[12], 0.707106769f, t);
          pfma(dyv[14], -0.456435472f, t);
        }
        const EVec d12_53 = dms[53 * NQV];
        const float4 a14 = *reinterpret_cast<const float4*>(As + 56);
        pfma(u12_1, a14.x, d12_53);
        { const float2 t = pmul(sx12_1, d12_53);
          pfma(dyv[13], 0.456435472f, t);
          pfma(dyv[15], -0.353553385f, t);
        }
        const EVec d12_54 = dms[54 * NQV];
        pfma(u12_1, a14.w, d12_54);
        { const float2 t = pmul(sx12_1, d12_54);
          pfma(dyv[14], 0.353553385f, t);
        }
        pfma(u12_2, a10.w, d12_48);
        { const float2 t = pmul(sx12_2, d12_48);
          pfma(dyv[15], 0.866025388f, t);
        }
        pfma(u12_2, a11.z, d12_49);
        { const float2 t = pmul(sx12_2, d12_49);
          pfma(dyv[14], 0.577350259f, t);
        }
        pfma(u12_2, a12.y, d12_50);
        { const float2 t = pmul(sx12_2, d12_50);
          pfma(dyv[13], 0.288675129f, t);
        }
        pfma(u12_3, a13.x, d12_51);
        { const float2 t = pmul(sx12_3, d12_51);
          pfma(dyv[11], 0.707106769f, t);
        }
        pfma(u12_2, a13.z, d12_52);
        { const float2 t = pmul(sx12_2, d12_52);
          pfma(dyv[11], -0.288675129f, t);
        }
        pfma(u12_2, a14.y, d12_53);
        { const float2 t = pmul(sx12_2, d12_53);
          pfma(dyv[10], -0.577350259f, t);
        }
        const float4 a15 = *reinterpret_cast<const float4*>(As + 60);
        pfma(u12_2, a15.x, d12_54);
        { const float2 t = pmul(sx12_2, d12_54);
          pfma(dyv[9], -0.866025388f, t);
        }
        pfma(u12_3, a11.x, d12_48);
        { const float2 t = pmul(sx12_3, d12_48);
          pfma(dyv[14], -0.353553385f, t);
        }
        pfma(u12_3, a11.w, d12_49);
        { const float2 t = pmul(sx12_3, d12_49);
          pfma(dyv[13], -0.456435472f, t);
          pfma(dyv[15], -0.353553385f, t);
        }
        pfma(u12_3, a12.z, d12_50);
        { const float2 t = pmul(sx12_3, d12_50);
          pfma(dyv[12], -0.707106769f, t);
          pfma(dyv[14], -0.456435472f, t);
        }
        pfma(u12_3, a13.w, d12_52);
        { const float2 t = pmul(sx12_3, d12_52);
          pfma(dyv[10], 0.456435472f, t);
        }
        pfma(u12_3, a14.z, d12_53);
        { const float2 t = pmul(sx12_3, d12_53);
          pfma(dyv[9], 0.353553385f, t);
          pfma(dyv[11], 0.456435472f, t);
        }
        pfma(u12_3, a15.y, d12_54);
        { const float2 t = pmul(sx12_3, d12_54);
          pfma(dyv[10], 0.353553385f, t);
        }
        EVec ds12 = pmul(x1, u12_1);
        pfma(ds12, x2, u12_2);
        pfma(ds12, x3, u12_3);
        if (gw) gw[12 * NQV] = ds12;
        pfma(dxp[1], s12, u12_1);
        pfma(dxp[2], s12, u12_2);
        pfma(dxp[3], s12, u12_3);
        dyl[0] = dyv[0].x + dyv[0].y;
        dyl[1] = dyv[1].x + dyv[1].y;
        dyl[2] = dyv[2].x + dyv[2].y;
        dyl[3] = dyv[3].x + dyv[3].y;
        dyl[4] = dyv[4].x + dyv[4].y;
        dyl[5] = dyv[5].x + dyv[5].y;
        dyl[6] = dyv[6].x + dyv[6].y;
        dyl[7] = dyv[7].x + dyv[7].y;
        dyl[8] = dyv[8].x + dyv[8].y;
        dyl[9] = dyv[9].x + dyv[9].y;
        dyl[10] = dyv[10].x + dyv[10].y;
        dyl[11] = dyv[11].x + dyv[11].y;
        dyl[12] = dyv[12].x + dyv[12].y;
        dyl[13] = dyv[13].x + dyv[13].y;
        dyl[14] = dyv[14].x + dyv[14].y;
        dyl[15] = dyv[15].x + dyv[15].y;
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
        const float4 a8 = *reinterpret_cast<const float4*>(As + 32);
        const float4 b8 = *reinterpret_cast<const float4*>(Bs + 32);
        pfma(v1_1, a8.x, d1_1);
        pfma(w1_1, b8.x, d1_1);
        { const float t = vdot(sxu1_1, d1_1);
          dyl[1] = 0.577350259f * t;
        }
        pfma(v1_2, a8.y, d1_1);
        pfma(w1_2, b8.y, d1_1);
        { const float t = vdot(sxu1_2, d1_1);
          dyl[2] = 0.577350259f * t;
        }
        pfma(v1_3, a8.z, d1_1);
        pfma(w1_3, b8.z, d1_1);
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
        pfma(v2_0, a0.y, d2_2);
        pfma(w2_0, b0.y, d2_2);
        { const float t = vdot(sxu2_0, d2_2);
          dyl[1] = fmaf(1.0f, t, dyl[1]);
        }
        const DVec d2_3 = dms[3 * NQV];
        pfma(v2_0, a0.z, d2_3);
        pfma(w2_0, b0.z, d2_3);
        { const float t = vdot(sxu2_0, d2_3);
          dyl[2] = fmaf(1.0f, t, dyl[2]);
        }
        const DVec d2_4 = dms[4 * NQV];
        pfma(v2_0, a0.w, d2_4);
        pfma(w2_0, b0.w, d2_4);
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
        const float4 a16 = *reinterpret_cast<const float4*>(As + 64);
        const float4 b16 = *reinterpret_cast<const float4*>(Bs + 64);
        pfma(v3_1, a16.x, d3_5);
        pfma(w3_1, b16.x, d3_5);
        { const float t = vdot(sxu3_1, d3_5);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        const DVec d3_6 = dms[6 * NQV];
        pfma(v3_2, a16.y, d3_6);
        pfma(w3_2, b16.y, d3_6);
        { const float t = vdot(sxu3_2, d3_6);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        const DVec d3_7 = dms[7 * NQV];
        pfma(v3_3, a16.z, d3_7);
        pfma(w3_3, b16.z, d3_7);
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
        const float4 a23 = *reinterpret_cast<const float4*>(As + 92);
        const float4 b23 = *reinterpret_cast<const float4*>(Bs + 92);
        pfma(v4_1, a23.x, d4_8);
        pfma(w4_1, b23.x, d4_8);
        { const float t = vdot(sxu4_1, d4_8);
          dyl[6] = 0.316227764f * t;
          dyl[8] = 0.547722578f * t;
        }
        const DVec d4_9 = dms[9 * NQV];
        pfma(v4_1, a23.w, d4_9);
        pfma(w4_1, b23.w, d4_9);
        { const float t = vdot(sxu4_1, d4_9);
          dyl[5] = -0.547722578f * t;
        }
        const DVec d4_10 = dms[10 * NQV];
        const float4 a24 = *reinterpret_cast<const float4*>(As + 96);
        const float4 b24 = *reinterpret_cast<const float4*>(Bs + 96);
        pfma(v4_1, a24.z, d4_10);
        pfma(w4_1, b24.z, d4_10);
        { const float t = vdot(sxu4_1, d4_10);
          dyl[4] = -0.547722578f * t;
        }
        pfma(v4_2, a23.y, d4_8);
        pfma(w4_2, b23.y, d4_8);
        { const float t = vdot(sxu4_2, d4_8);
          dyl[5] = fmaf(-0.547722578f, t, dyl[5]);
        }
        pfma(v4_2, a24.x, d4_9);
        pfma(w4_2, b24.x, d4_9);
        { const float t = vdot(sxu4_2, d4_9);
          dyl[6] = fmaf(-0.632455528f, t, dyl[6]);
        }
        pfma(v4_2, a24.w, d4_10);
        pfma(w4_2, b24.w, d4_10);
        { const float t = vdot(sxu4_2, d4_10);
          dyl[7] = -0.547722578f * t;
        }
        pfma(v4_3, a23.z, d4_8);
        pfma(w4_3, b23.z, d4_8);
        { const float t = vdot(sxu4_3, d4_8);
          dyl[4] = fmaf(-0.547722578f, t, dyl[4]);
        }
        pfma(v4_3, a24.y, d4_9);
        pfma(w4_3, b24.y, d4_9);
        { const float t = vdot(sxu4_3, d4_9);
          dyl[7] = fmaf(-0.547722578f, t, dyl[7]);
        }
        const float4 a25 = *reinterpret_cast<const float4*>(As + 100);
        const float4 b25 = *reinterpret_cast<const float4*>(Bs + 100);
        pfma(v4_3, a25.x, d4_10);
        pfma(w4_3, b25.x, d4_10);
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
        const DVec s5 = ss[5 * NQV];  // path 5: l1=1 l2=1 -> L=1
        const DVec us5 = uss[5 * NQV];
        DVec sxu5_1 = pmul(s5, ux1); pfma(sxu5_1, us5, x1);
        DVec v5_1; vzero(v5_1);
        DVec w5_1; vzero(w5_1);
        DVec sxu5_2 = pmul(s5, ux2); pfma(sxu5_2, us5, x2);
        DVec v5_2; vzero(v5_2);
        DVec w5_2; vzero(w5_2);
        DVec sxu5_3 = pmul(s5, ux3); pfma(sxu5_3, us5, x3);
        DVec v5_3; vzero(v5_3);
        DVec w5_3; vzero(w5_3);
        const DVec d5_11 = dms[11 * NQV];
        pfma(v5_2, a16.w, d5_11);
        pfma(w5_2, b16.w, d5_11);
        { const float t = vdot(sxu5_2, d5_11);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        const DVec d5_12 = dms[12 * NQV];
        const float4 a17 = *reinterpret_cast<const float4*>(As + 68);
        const float4 b17 = *reinterpret_cast<const float4*>(Bs + 68);
        pfma(v5_1, a17.y, d5_12);
        pfma(w5_1, b17.y, d5_12);
        { const float t = vdot(sxu5_1, d5_12);
          dyl[3] = fmaf(-0.707106769f, t, dyl[3]);
        }
        const DVec d5_13 = dms[13 * NQV];
        pfma(v5_1, a17.w, d5_13);
        pfma(w5_1, b17.w, d5_13);
        { const float t = vdot(sxu5_1, d5_13);
          dyl[2] = fmaf(0.707106769f, t, dyl[2]);
        }
        pfma(v5_3, a17.x, d5_11);
        pfma(w5_3, b17.x, d5_11);
        { const float t = vdot(sxu5_3, d5_11);
          dyl[2] = fmaf(-0.707106769f, t, dyl[2]);
        }
        pfma(v5_3, a17.z, d5_12);
        pfma(w5_3, b17.z, d5_12);
        { const float t = vdot(sxu5_3, d5_12);
          dyl[1] = fmaf(0.707106769f, t, dyl[1]);
        }
        const float4 a18 = *reinterpret_cast<const float4*>(As + 72);
        const float4 b18 = *reinterpret_cast<const float4*>(Bs + 72);
        pfma(v5_2, a18.x, d5_13);
        pfma(w5_2, b18.x, d5_13);
        { const float t = vdot(sxu5_2, d5_13);
          dyl[1] = fmaf(-0.707106769f, t, dyl[1]);
        }
        DVec ds5 = pmul(ux1, v5_1); pfma(ds5, x1, w5_1);
        pfma(ds5, ux2, v5_2); pfma(ds5, x2, w5_2);
        pfma(ds5, ux3, v5_3); pfma(ds5, x3, w5_3);
        if (gw) gw[5 * NQV] = ds5;
        pfma(dxp[1], us5, v5_1); pfma(dxp[1], s5, w5_1);
        pfma(dxp[2], us5, v5_2); pfma(dxp[2], s5, w5_2);
        pfma(dxp[3], us5, v5_3); pfma(dxp[3], s5, w5_3);
        const DVec s6 = ss[6 * NQV];  // path 6: l1=0 l2=2 -> L=2
        const DVec us6 = uss[6 * NQV];
        DVec sxu6_0 = pmul(s6, ux0); pfma(sxu6_0, us6, x0);
        DVec v6_0; vzero(v6_0);
        DVec w6_0; vzero(w6_0);
        const DVec d6_14 = dms[14 * NQV];
        pfma(v6_0, a25.y, d6_14);
        pfma(w6_0, b25.y, d6_14);
        { const float t = vdot(sxu6_0, d6_14);
          dyl[4] = fmaf(1.0f, t, dyl[4]);
        }
        const DVec d6_15 = dms[15 * NQV];
        pfma(v6_0, a25.z, d6_15);
        pfma(w6_0, b25.z, d6_15);
        { const float t = vdot(sxu6_0, d6_15);
          dyl[5] = fmaf(1.0f, t, dyl[5]);
        }
        const DVec d6_16 = dms[16 * NQV];
        pfma(v6_0, a25.w, d6_16);
        pfma(w6_0, b25.w, d6_16);
        { const float t = vdot(sxu6_0, d6_16);
          dyl[6] = fmaf(1.0f, t, dyl[6]);
        }
        const DVec d6_17 = dms[17 * NQV];
        const float4 a26 = *reinterpret_cast<const float4*>(As + 104);
        const float4 b26 = *reinterpret_cast<const float4*>(Bs + 104);
        pfma(v6_0, a26.x, d6_17);
        pfma(w6_0, b26.x, d6_17);
        { const float t = vdot(sxu6_0, d6_17);
          dyl[7] = fmaf(1.0f, t, dyl[7]);
        }
        const DVec d6_18 = dms[18 * NQV];
        pfma(v6_0, a26.y, d6_18);
        pfma(w6_0, b26.y, d6_18);
        { const float t = vdot(sxu6_0, d6_18);
          dyl[8] = fmaf(1.0f, t, dyl[8]);
        }
        DVec ds6 = pmul(ux0, v6_0); pfma(ds6, x0, w6_0);
        if (gw) gw[6 * NQV] = ds6;
        pfma(dxp[0], us6, v6_0); pfma(dxp[0], s6, w6_0);
        const DVec s7 = ss[7 * NQV];  // path 7: l1=1 l2=1 -> L=2
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
        const DVec d7_19 = dms[19 * NQV];
        const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
        const float4 b1 = *reinterpret_cast<const float4*>(Bs + 4);
        pfma(v7_1, a1.x, d7_19);
        pfma(w7_1, b1.x, d7_19);
        { const float t = vdot(sxu7_1, d7_19);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        const DVec d7_20 = dms[20 * NQV];
        pfma(v7_1, a1.z, d7_20);
        pfma(w7_1, b1.z, d7_20);
        { const float t = vdot(sxu7_1, d7_20);
          dyl[2] = fmaf(0.707106769f, t, dyl[2]);
        }
        const DVec d7_21 = dms[21 * NQV];
        const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
        const float4 b2 = *reinterpret_cast<const float4*>(Bs + 8);
        pfma(v7_1, a2.x, d7_21);
        pfma(w7_1, b2.x, d7_21);
        { const float t = vdot(sxu7_1, d7_21);
          dyl[1] = fmaf(-0.408248305f, t, dyl[1]);
        }
        const DVec d7_22 = dms[22 * NQV];
        pfma(v7_2, a2.w, d7_22);
        pfma(w7_2, b2.w, d7_22);
        { const float t = vdot(sxu7_2, d7_22);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        const DVec d7_23 = dms[23 * NQV];
        const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
        const float4 b3 = *reinterpret_cast<const float4*>(Bs + 12);
        pfma(v7_1, a3.y, d7_23);
        pfma(w7_1, b3.y, d7_23);
        { const float t = vdot(sxu7_1, d7_23);
          dyl[1] = fmaf(-0.707106769f, t, dyl[1]);
        }
        pfma(v7_3, a1.y, d7_19);
        pfma(w7_3, b1.y, d7_19);
        { const float t = vdot(sxu7_3, d7_19);
          dyl[1] = fmaf(0.707106769f, t, dyl[1]);
        }
        pfma(v7_2, a1.w, d7_20);
        pfma(w7_2, b1.w, d7_20);
        { const float t = vdot(sxu7_2, d7_20);
          dyl[1] = fmaf(0.707106769f, t, dyl[1]);
        }
        pfma(v7_2, a2.y, d7_21);
        pfma(w7_2, b2.y, d7_21);
        { const float t = vdot(sxu7_2, d7_21);
          dyl[2] = fmaf(0.816496611f, t, dyl[2]);
        }
        pfma(v7_3, a3.x, d7_22);
        pfma(w7_3, b3.x, d7_22);
        { const float t = vdot(sxu7_3, d7_22);
          dyl[2] = fmaf(0.707106769f, t, dyl[2]);
        }
        pfma(v7_3, a3.z, d7_23);
        pfma(w7_3, b3.z, d7_23);
        { const float t = vdot(sxu7_3, d7_23);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        pfma(v7_3, a2.z, d7_21);
        pfma(w7_3, b2.z, d7_21);
        { const float t = vdot(sxu7_3, d7_21);
          dyl[3] = fmaf(-0.408248305f, t, dyl[3]);
        }
        DVec ds7 = pmul(ux1, v7_1); pfma(ds7, x1, w7_1);
        pfma(ds7, ux2, v7_2); pfma(ds7, x2, w7_2);
        pfma(ds7, ux3, v7_3); pfma(ds7, x3, w7_3);
        if (gw) gw[7 * NQV] = ds7;
        pfma(dxp[1], us7, v7_1); pfma(dxp[1], s7, w7_1);
        pfma(dxp[2], us7, v7_2); pfma(dxp[2], s7, w7_2);
        pfma(dxp[3], us7, v7_3); pfma(dxp[3], s7, w7_3);
        const DVec s8 = ss[8 * NQV];  // path 8: l1=1 l2=3 -> L=2
        const DVec us8 = uss[8 * NQV];
        DVec sxu8_1 = pmul(s8, ux1); pfma(sxu8_1, us8, x1);
        DVec v8_1; vzero(v8_1);
        DVec w8_1; vzero(w8_1);
        DVec sxu8_2 = pmul(s8, ux2); pfma(sxu8_2, us8, x2);
        DVec v8_2; vzero(v8_2);
        DVec w8_2; vzero(w8_2);
        DVec sxu8_3 = pmul(s8, ux3); pfma(sxu8_3, us8, x3);
        DVec v8_3; vzero(v8_3);
        DVec w8_3; vzero(w8_3);
        const DVec d8_24 = dms[24 * NQV];
        pfma(v8_1, a26.z, d8_24);
        pfma(w8_1, b26.z, d8_24);
        { const float t = vdot(sxu8_1, d8_24);
          dyl[13] = 0.154303357f * t;
          dyl[15] = 0.597614288f * t;
        }
        const DVec d8_25 = dms[25 * NQV];
        const float4 a27 = *reinterpret_cast<const float4*>(As + 108);
        const float4 b27 = *reinterpret_cast<const float4*>(Bs + 108);
        pfma(v8_1, a27.y, d8_25);
        pfma(w8_1, b27.y, d8_25);
        { const float t = vdot(sxu8_1, d8_25);
          dyl[12] = 0.377964467f * t;
          dyl[14] = 0.487950027f * t;
        }
        const DVec d8_26 = dms[26 * NQV];
        const float4 a28 = *reinterpret_cast<const float4*>(As + 112);
        const float4 b28 = *reinterpret_cast<const float4*>(Bs + 112);
        pfma(v8_1, a28.x, d8_26);
        pfma(w8_1, b28.x, d8_26);
        { const float t = vdot(sxu8_1, d8_26);
          dyl[11] = -0.534522474f * t;
        }
        const DVec d8_27 = dms[27 * NQV];
        pfma(v8_1, a28.w, d8_27);
        pfma(w8_1, b28.w, d8_27);
        { const float t = vdot(sxu8_1, d8_27);
          dyl[10] = -0.487950027f * t;
        }
        const DVec d8_28 = dms[28 * NQV];
        const float4 a29 = *reinterpret_cast<const float4*>(As + 116);
        const float4 b29 = *reinterpret_cast<const float4*>(Bs + 116);
        pfma(v8_1, a29.z, d8_28);
        pfma(w8_1, b29.z, d8_28);
        { const float t = vdot(sxu8_1, d8_28);
          dyl[9] = -0.597614288f * t;
          dyl[11] = fmaf(-0.154303357f, t, dyl[11]);
        }
        pfma(v8_2, a26.w, d8_24);
        pfma(w8_2, b26.w, d8_24);
        { const float t = vdot(sxu8_2, d8_24);
          dyl[10] = fmaf(-0.487950027f, t, dyl[10]);
        }
        pfma(v8_2, a27.z, d8_25);
        pfma(w8_2, b27.z, d8_25);
        { const float t = vdot(sxu8_2, d8_25);
          dyl[11] = fmaf(-0.617213428f, t, dyl[11]);
        }
        pfma(v8_2, a28.y, d8_26);
        pfma(w8_2, b28.y, d8_26);
        { const float t = vdot(sxu8_2, d8_26);
          dyl[12] = fmaf(-0.654653668f, t, dyl[12]);
        }
        pfma(v8_2, a29.x, d8_27);
        pfma(w8_2, b29.x, d8_27);
        { const float t = vdot(sxu8_2, d8_27);
          dyl[13] = fmaf(-0.617213428f, t, dyl[13]);
        }
        pfma(v8_2, a29.w, d8_28);
        pfma(w8_2, b29.w, d8_28);
        { const float t = vdot(sxu8_2, d8_28);
          dyl[14] = fmaf(-0.487950027f, t, dyl[14]);
        }
        pfma(v8_3, a27.x, d8_24);
        pfma(w8_3, b27.x, d8_24);
        { const float t = vdot(sxu8_3, d8_24);
          dyl[9] = fmaf(-0.597614288f, t, dyl[9]);
          dyl[11] = fmaf(0.154303357f, t, dyl[11]);
        }
        pfma(v8_3, a27.w, d8_25);
        pfma(w8_3, b27.w, d8_25);
        { const float t = vdot(sxu8_3, d8_25);
          dyl[10] = fmaf(-0.487950027f, t, dyl[10]);
        }
        pfma(v8_3, a28.z, d8_26);
        pfma(w8_3, b28.z, d8_26);
        { const float t = vdot(sxu8_3, d8_26);
          dyl[13] = fmaf(-0.534522474f, t, dyl[13]);
        }
        pfma(v8_3, a29.y, d8_27);
        pfma(w8_3, b29.y, d8_27);
        { const float t = vdot(sxu8_3, d8_27);
          dyl[12] = fmaf(0.377964467f, t, dyl[12]);
          dyl[14] = fmaf(-0.487950027f, t, dyl[14]);
        }
        const float4 a30 = *reinterpret_cast<const float4*>(As + 120);
        const float4 b30 = *reinterpret_cast<const float4*>(Bs + 120);
        pfma(v8_3, a30.x, d8_28);
        pfma(w8_3, b30.x, d8_28);
        { const float t = vdot(sxu8_3, d8_28);
          dyl[13] = fmaf(0.154303357f, t, dyl[13]);
          dyl[15] = fmaf(-0.597614288f, t, dyl[15]);
        }
        DVec ds8 = pmul(ux1, v8_1); pfma(ds8, x1, w8_1);
        pfma(ds8, ux2, v8_2); pfma(ds8, x2, w8_2);
        pfma(ds8, ux3, v8_3); pfma(ds8, x3, w8_3);
        if (gw) gw[8 * NQV] = ds8;
        pfma(dxp[1], us8, v8_1); pfma(dxp[1], s8, w8_1);
        pfma(dxp[2], us8, v8_2); pfma(dxp[2], s8, w8_2);
        pfma(dxp[3], us8, v8_3); pfma(dxp[3], s8, w8_3);
        const DVec s9 = ss[9 * NQV];  // path 9: l1=1 l2=2 -> L=2
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
        const DVec d9_29 = dms[29 * NQV];
        pfma(v9_1, a3.w, d9_29);
        pfma(w9_1, b3.w, d9_29);
        { const float t = vdot(sxu9_1, d9_29);
          dyl[5] = fmaf(0.408248305f, t, dyl[5]);
        }
        const DVec d9_30 = dms[30 * NQV];
        const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
        const float4 b4 = *reinterpret_cast<const float4*>(Bs + 16);
        pfma(v9_1, a4.z, d9_30);
        pfma(w9_1, b4.z, d9_30);
        { const float t = vdot(sxu9_1, d9_30);
          dyl[4] = fmaf(-0.408248305f, t, dyl[4]);
        }
        const DVec d9_31 = dms[31 * NQV];
        const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
        const float4 b5 = *reinterpret_cast<const float4*>(Bs + 20);
        pfma(v9_1, a5.y, d9_31);
        pfma(w9_1, b5.y, d9_31);
        { const float t = vdot(sxu9_1, d9_31);
          dyl[7] = fmaf(-0.707106769f, t, dyl[7]);
        }
        const DVec d9_32 = dms[32 * NQV];
        pfma(v9_1, a5.w, d9_32);
        pfma(w9_1, b5.w, d9_32);
        { const float t = vdot(sxu9_1, d9_32);
          dyl[6] = fmaf(0.707106769f, t, dyl[6]);
          dyl[8] = fmaf(-0.408248305f, t, dyl[8]);
        }
        const DVec d9_33 = dms[33 * NQV];
        const float4 a6 = *reinterpret_cast<const float4*>(As + 24);
        const float4 b6 = *reinterpret_cast<const float4*>(Bs + 24);
        pfma(v9_1, a6.z, d9_33);
        pfma(w9_1, b6.z, d9_33);
        { const float t = vdot(sxu9_1, d9_33);
          dyl[7] = fmaf(0.408248305f, t, dyl[7]);
        }
        pfma(v9_2, a4.x, d9_29);
        pfma(w9_2, b4.x, d9_29);
        { const float t = vdot(sxu9_2, d9_29);
          dyl[8] = fmaf(0.816496611f, t, dyl[8]);
        }
        pfma(v9_2, a4.w, d9_30);
        pfma(w9_2, b4.w, d9_30);
        { const float t = vdot(sxu9_2, d9_30);
          dyl[7] = fmaf(0.408248305f, t, dyl[7]);
        }
        pfma(v9_3, a5.z, d9_31);
        pfma(w9_3, b5.z, d9_31);
        { const float t = vdot(sxu9_3, d9_31);
          dyl[5] = fmaf(0.707106769f, t, dyl[5]);
        }
        pfma(v9_2, a6.x, d9_32);
        pfma(w9_2, b6.x, d9_32);
        { const float t = vdot(sxu9_2, d9_32);
          dyl[5] = fmaf(-0.408248305f, t, dyl[5]);
        }
        pfma(v9_2, a6.w, d9_33);
        pfma(w9_2, b6.w, d9_33);
        { const float t = vdot(sxu9_2, d9_33);
          dyl[4] = fmaf(-0.816496611f, t, dyl[4]);
        }
        pfma(v9_3, a4.y, d9_29);
        pfma(w9_3, b4.y, d9_29);
        { const float t = vdot(sxu9_3, d9_29);
          dyl[7] = fmaf(-0.408248305f, t, dyl[7]);
        }
        pfma(v9_3, a5.x, d9_30);
        pfma(w9_3, b5.x, d9_30);
        { const float t = vdot(sxu9_3, d9_30);
          dyl[6] = fmaf(-0.707106769f, t, dyl[6]);
          dyl[8] = fmaf(-0.408248305f, t, dyl[8]);
        }
        pfma(v9_3, a6.y, d9_32);
        pfma(w9_3, b6.y, d9_32);
        { const float t = vdot(sxu9_3, d9_32);
          dyl[4] = fmaf(0.408248305f, t, dyl[4]);
        }
        const float4 a7 = *reinterpret_cast<const float4*>(As + 28);
        const float4 b7 = *reinterpret_cast<const float4*>(Bs + 28);
        pfma(v9_3, a7.x, d9_33);
        pfma(w9_3, b7.x, d9_33);
        { const float t = vdot(sxu9_3, d9_33);
          dyl[5] = fmaf(0.408248305f, t, dyl[5]);
        }
        DVec ds9 = pmul(ux1, v9_1); pfma(ds9, x1, w9_1);
        pfma(ds9, ux2, v9_2); pfma(ds9, x2, w9_2);
        pfma(ds9, ux3, v9_3); pfma(ds9, x3, w9_3);
        if (gw) gw[9 * NQV] = ds9;
        pfma(dxp[1], us9, v9_1); pfma(dxp[1], s9, w9_1);
        pfma(dxp[2], us9, v9_2); pfma(dxp[2], s9, w9_2);
        pfma(dxp[3], us9, v9_3); pfma(dxp[3], s9, w9_3);
        const DVec s10 = ss[10 * NQV];  // path 10: l1=0 l2=3 -> L=3
        const DVec us10 = uss[10 * NQV];
        DVec sxu10_0 = pmul(s10, ux0); pfma(sxu10_0, us10, x0);
        DVec v10_0; vzero(v10_0);
        DVec w10_0; vzero(w10_0);
        const DVec d10_34 = dms[34 * NQV];
        pfma(v10_0, a8.w, d10_34);
        pfma(w10_0, b8.w, d10_34);
        { const float t = vdot(sxu10_0, d10_34);
          dyl[9] = fmaf(1.0f, t, dyl[9]);
        }
        const DVec d10_35 = dms[35 * NQV];
        const float4 a9 = *reinterpret_cast<const float4*>(As + 36);
        const float4 b9 = *reinterpret_cast<const float4*>(Bs + 36);
        pfma(v10_0, a9.x, d10_35);
        pfma(w10_0, b9.x, d10_35);
        { const float t = vdot(sxu10_0, d10_35);
          dyl[10] = fmaf(1.0f, t, dyl[10]);
        }
        const DVec d10_36 = dms[36 * NQV];
        pfma(v10_0, a9.y, d10_36);
        pfma(w10_0, b9.y, d10_36);
        { const float t = vdot(sxu10_0, d10_36);
          dyl[11] = fmaf(1.0f, t, dyl[11]);
        }
        const DVec d10_37 = dms[37 * NQV];
        pfma(v10_0, a9.z, d10_37);
        pfma(w10_0, b9.z, d10_37);
        { const float t = vdot(sxu10_0, d10_37);
          dyl[12] = fmaf(1.0f, t, dyl[12]);
        }
        const DVec d10_38 = dms[38 * NQV];
        pfma(v10_0, a9.w, d10_38);
        pfma(w10_0, b9.w, d10_38);
        { const float t = vdot(sxu10_0, d10_38);
          dyl[13] = fmaf(1.0f, t, dyl[13]);
        }
        const DVec d10_39 = dms[39 * NQV];
        const float4 a10 = *reinterpret_cast<const float4*>(As + 40);
        const float4 b10 = *reinterpret_cast<const float4*>(Bs + 40);
        pfma(v10_0, a10.x, d10_39);
        pfma(w10_0, b10.x, d10_39);
        { const float t = vdot(sxu10_0, d10_39);
          dyl[14] = fmaf(1.0f, t, dyl[14]);
        }
        const DVec d10_40 = dms[40 * NQV];
        pfma(v10_0, a10.y, d10_40);
        pfma(w10_0, b10.y, d10_40);
        { const float t = vdot(sxu10_0, d10_40);
          dyl[15] = fmaf(1.0f, t, dyl[15]);
        }
        DVec ds10 = pmul(ux0, v10_0); pfma(ds10, x0, w10_0);
        if (gw) gw[10 * NQV] = ds10;
        pfma(dxp[0], us10, v10_0); pfma(dxp[0], s10, w10_0);
        const DVec s11 = ss[11 * NQV];  // path 11: l1=1 l2=2 -> L=3
        const DVec us11 = uss[11 * NQV];
        DVec sxu11_1 = pmul(s11, ux1); pfma(sxu11_1, us11, x1);
        DVec v11_1; vzero(v11_1);
        DVec w11_1; vzero(w11_1);
        DVec sxu11_2 = pmul(s11, ux2); pfma(sxu11_2, us11, x2);
        DVec v11_2; vzero(v11_2);
        DVec w11_2; vzero(w11_2);
        DVec sxu11_3 = pmul(s11, ux3); pfma(sxu11_3, us11, x3);
        DVec v11_3; vzero(v11_3);
        DVec w11_3; vzero(w11_3);
        const DVec d11_41 = dms[41 * NQV];
        pfma(v11_1, a18.y, d11_41);
        pfma(w11_1, b18.y, d11_41);
        { const float t = vdot(sxu11_1, d11_41);
          dyl[8] = fmaf(0.707106769f, t, dyl[8]);
        }
        const DVec d11_42 = dms[42 * NQV];
        pfma(v11_1, a18.w, d11_42);
        pfma(w11_1, b18.w, d11_42);
        { const float t = vdot(sxu11_1, d11_42);
          dyl[7] = fmaf(0.577350259f, t, dyl[7]);
        }
        const DVec d11_43 = dms[43 * NQV];
        const float4 a19 = *reinterpret_cast<const float4*>(As + 76);
        const float4 b19 = *reinterpret_cast<const float4*>(Bs + 76);
        pfma(v11_1, a19.z, d11_43);
        pfma(w11_1, b19.z, d11_43);
        { const float t = vdot(sxu11_1, d11_43);
          dyl[6] = fmaf(0.632455528f, t, dyl[6]);
          dyl[8] = fmaf(0.182574183f, t, dyl[8]);
        }
        const DVec d11_44 = dms[44 * NQV];
        const float4 a20 = *reinterpret_cast<const float4*>(As + 80);
        const float4 b20 = *reinterpret_cast<const float4*>(Bs + 80);
        pfma(v11_1, a20.y, d11_44);
        pfma(w11_1, b20.y, d11_44);
        { const float t = vdot(sxu11_1, d11_44);
          dyl[5] = fmaf(-0.44721359f, t, dyl[5]);
        }
        const DVec d11_45 = dms[45 * NQV];
        const float4 a21 = *reinterpret_cast<const float4*>(As + 84);
        const float4 b21 = *reinterpret_cast<const float4*>(Bs + 84);
        pfma(v11_1, a21.x, d11_45);
        pfma(w11_1, b21.x, d11_45);
        { const float t = vdot(sxu11_1, d11_45);
          dyl[4] = fmaf(-0.182574183f, t, dyl[4]);
        }
        const DVec d11_46 = dms[46 * NQV];
        pfma(v11_1, a21.w, d11_46);
        pfma(w11_1, b21.w, d11_46);
        { const float t = vdot(sxu11_1, d11_46);
          dyl[5] = fmaf(-0.577350259f, t, dyl[5]);
        }
        const DVec d11_47 = dms[47 * NQV];
        const float4 a22 = *reinterpret_cast<const float4*>(As + 88);
        const float4 b22 = *reinterpret_cast<const float4*>(Bs + 88);
        pfma(v11_1, a22.z, d11_47);
        pfma(w11_1, b22.z, d11_47);
        { const float t = vdot(sxu11_1, d11_47);
          dyl[4] = fmaf(-0.707106769f, t, dyl[4]);
        }
        pfma(v11_3, a18.z, d11_41);
        pfma(w11_3, b18.z, d11_41);
        { const float t = vdot(sxu11_3, d11_41);
          dyl[4] = fmaf(0.707106769f, t, dyl[4]);
        }
        pfma(v11_2, a19.x, d11_42);
        pfma(w11_2, b19.x, d11_42);
        { const float t = vdot(sxu11_2, d11_42);
          dyl[4] = fmaf(0.577350259f, t, dyl[4]);
        }
        pfma(v11_2, a19.w, d11_43);
        pfma(w11_2, b19.w, d11_43);
        { const float t = vdot(sxu11_2, d11_43);
          dyl[5] = fmaf(0.730296731f, t, dyl[5]);
        }
        pfma(v11_2, a20.z, d11_44);
        pfma(w11_2, b20.z, d11_44);
        { const float t = vdot(sxu11_2, d11_44);
          dyl[6] = fmaf(0.774596691f, t, dyl[6]);
        }
        pfma(v11_2, a21.y, d11_45);
        pfma(w11_2, b21.y, d11_45);
        { const float t = vdot(sxu11_2, d11_45);
          dyl[7] = fmaf(0.730296731f, t, dyl[7]);
        }
        pfma(v11_2, a22.x, d11_46);
        pfma(w11_2, b22.x, d11_46);
        { const float t = vdot(sxu11_2, d11_46);
          dyl[8] = fmaf(0.577350259f, t, dyl[8]);
        }
        pfma(v11_3, a22.w, d11_47);
        pfma(w11_3, b22.w, d11_47);
        { const float t = vdot(sxu11_3, d11_47);
          dyl[8] = fmaf(0.707106769f, t, dyl[8]);
        }
        pfma(v11_3, a19.y, d11_42);
        pfma(w11_3, b19.y, d11_42);
        { const float t = vdot(sxu11_3, d11_42);
          dyl[5] = fmaf(0.577350259f, t, dyl[5]);
        }
        pfma(v11_3, a20.x, d11_43);
        pfma(w11_3, b20.x, d11_43);
        { const float t = vdot(sxu11_3, d11_43);
          dyl[4] = fmaf(-0.182574183f, t, dyl[4]);
        }
        pfma(v11_3, a20.w, d11_44);
        pfma(w11_3, b20.w, d11_44);
        { const float t = vdot(sxu11_3, d11_44);
          dyl[7] = fmaf(-0.44721359f, t, dyl[7]);
        }
        pfma(v11_3, a21.z, d11_45);
        pfma(w11_3, b21.z, d11_45);
        { const float t = vdot(sxu11_3, d11_45);
          dyl[6] = fmaf(0.632455528f, t, dyl[6]);
          dyl[8] = fmaf(-0.182574183f, t, dyl[8]);
        }
        pfma(v11_3, a22.y, d11_46);
        pfma(w11_3, b22.y, d11_46);
        { const float t = vdot(sxu11_3, d11_46);
          dyl[7] = fmaf(0.577350259f, t, dyl[7]);
        }
        DVec ds11 = pmul(ux1, v11_1); pfma(ds11, x1, w11_1);
        pfma(ds11, ux2, v11_2); pfma(ds11, x2, w11_2);
        pfma(ds11, ux3, v11_3); pfma(ds11, x3, w11_3);
        if (gw) gw[11 * NQV] = ds11;
        pfma(dxp[1], us11, v11_1); pfma(dxp[1], s11, w11_1);
        pfma(dxp[2], us11, v11_2); pfma(dxp[2], s11, w11_2);
        pfma(dxp[3], us11, v11_3); pfma(dxp[3], s11, w11_3);
        const DVec s12 = ss[12 * NQV];  // path 12: l1=1 l2=3 -> L=3
        const DVec us12 = uss[12 * NQV];
        DVec sxu12_1 = pmul(s12, ux1); pfma(sxu12_1, us12, x1);
        DVec v12_1; vzero(v12_1);
        DVec w12_1; vzero(w12_1);
        DVec sxu12_2 = pmul(s12, ux2); pfma(sxu12_2, us12, x2);
        DVec v12_2; vzero(v12_2);
        DVec w12_2; vzero(w12_2);
        DVec sxu12_3 = pmul(s12, ux3); pfma(sxu12_3, us12, x3);
        DVec v12_3; vzero(v12_3);
        DVec w12_3; vzero(w12_3);
        const DVec d12_48 = dms[48 * NQV];
        pfma(v12_1, a10.z, d12_48);
        pfma(w12_1, b10.z, d12_48);
        { const float t = vdot(sxu12_1, d12_48);
          dyl[10] = fmaf(0.353553385f, t, dyl[10]);
        }
        const DVec d12_49 = dms[49 * NQV];
        const float4 a11 = *reinterpret_cast<const float4*>(As + 44);
        const float4 b11 = *reinterpret_cast<const float4*>(Bs + 44);
        pfma(v12_1, a11.y, d12_49);
        pfma(w12_1, b11.y, d12_49);
        { const float t = vdot(sxu12_1, d12_49);
          dyl[9] = fmaf(-0.353553385f, t, dyl[9]);
          dyl[11] = fmaf(0.456435472f, t, dyl[11]);
        }
        const DVec d12_50 = dms[50 * NQV];
        const float4 a12 = *reinterpret_cast<const float4*>(As + 48);
        const float4 b12 = *reinterpret_cast<const float4*>(Bs + 48);
        pfma(v12_1, a12.x, d12_50);
        pfma(w12_1, b12.x, d12_50);
        { const float t = vdot(sxu12_1, d12_50);
          dyl[10] = fmaf(-0.456435472f, t, dyl[10]);
        }
        const DVec d12_51 = dms[51 * NQV];
        pfma(v12_1, a12.w, d12_51);
        pfma(w12_1, b12.w, d12_51);
        { const float t = vdot(sxu12_1, d12_51);
          dyl[13] = fmaf(-0.707106769f, t, dyl[13]);
        }
        const DVec d12_52 = dms[52 * NQV];
        const float4 a13 = *reinterpret_cast<const float4*>(As + 52);
        const float4 b13 = *reinterpret_cast<const float4*>(Bs + 52);
        pfma(v12_1, a13.y, d12_52);
        pfma(w12_1, b13.y, d12_52);
        { const float t = vdot(sxu12_1, d12_52);
          dyl[12] = fmaf(0.707106769f, t, dyl[12]);
          dyl[14] = fmaf(-0.456435472f, t, dyl[14]);
        }
        const DVec d12_53 = dms[53 * NQV];
        const float4 a14 = *reinterpret_cast<const float4*>(As + 56);
        const float4 b14 = *reinterpret_cast<const float4*>(Bs + 56);
        pfma(v12_1, a14.x, d12_53);
        pfma(w12_1, b14.x, d12_53);
        { const float t = vdot(sxu12_1, d12_53);
          dyl[13] = fmaf(0.456435472f, t, dyl[13]);
          dyl[15] = fmaf(-0.353553385f, t, dyl[15]);
        }
        const DVec d12_54 = dms[54 * NQV];
        pfma(v12_1, a14.w, d12_54);
        pfma(w12_1, b14.w, d12_54);
        { const float t = vdot(sxu12_1, d12_54);
          dyl[14] = fmaf(0.353553385f, t, dyl[14]);
        }
        pfma(v12_2, a10.w, d12_48);
        pfma(w12_2, b10.w, d12_48);
        { const float t = vdot(sxu12_2, d12_48);
          dyl[15] = fmaf(0.866025388f, t, dyl[15]);
        }
        pfma(v12_2, a11.z, d12_49);
        pfma(w12_2, b11.z, d12_49);
        { const float t = vdot(sxu12_2, d12_49);
          dyl[14] = fmaf(0.577350259f, t, dyl[14]);
        }
        pfma(v12_2, a12.y, d12_50);
        pfma(w12_2, b12.y, d12_50);
        { const float t = vdot(sxu12_2, d12_50);
          dyl[13] = fmaf(0.288675129f, t, dyl[13]);
        }
        pfma(v12_3, a13.x, d12_51);
        pfma(w12_3, b13.x, d12_51);
        { const float t = vdot(sxu12_3, d12_51);
          dyl[11] = fmaf(0.707106769f, t, dyl[11]);
        }
        pfma(v12_2, a13.z, d12_52);
        pfma(w12_2, b13.z, d12_52);
        { const float t = vdot(sxu12_2, d12_52);
          dyl[11] = fmaf(-0.288675129f, t, dyl[11]);
        }
        pfma(v12_2, a14.y, d12_53);
        pfma(w12_2, b14.y, d12_53);
        { const float t = vdot(sxu12_2, d12_53);
          dyl[10] = fmaf(-0.577350259f, t, dyl[10]);
        }
        const float4 a15 = *reinterpret_cast<const float4*>(As + 60);
        const float4 b15 = *reinterpret_cast<const float4*>(Bs + 60);
        pfma(v12_2, a15.x, d12_54);
        pfma(w12_2, b15.x, d12_54);
        { const float t = vdot(sxu12_2, d12_54);
          dyl[9] = fmaf(-0.866025388f, t, dyl[9]);
        }
        pfma(v12_3, a11.x, d12_48);
        pfma(w12_3, b11.x, d12_48);
        { const float t = vdot(sxu12_3, d12_48);
          dyl[14] = fmaf(-0.353553385f, t, dyl[14]);
        }
        pfma(v12_3, a11.w, d12_49);
        pfma(w12_3, b11.w, d12_49);
        { const float t = vdot(sxu12_3, d12_49);
          dyl[13] = fmaf(-0.456435472f, t, dyl[13]);
          dyl[15] = fmaf(-0.353553385f, t, dyl[15]);
        }
        pfma(v12_3, a12.z, d12_50);
        pfma(w12_3, b12.z, d12_50);
        { const float t = vdot(sxu12_3, d12_50);
          dyl[12] = fmaf(-0.707106769f, t, dyl[12]);
          dyl[14] = fmaf(-0.456435472f, t, dyl[14]);
        }
        pfma(v12_3, a13.w, d12_52);
        pfma(w12_3, b13.w, d12_52);
        { const float t = vdot(sxu12_3, d12_52);
          dyl[10] = fmaf(0.456435472f, t, dyl[10]);
        }
        pfma(v12_3, a14.z, d12_53);
        pfma(w12_3, b14.z, d12_53);
        { const float t = vdot(sxu12_3, d12_53);
          dyl[9] = fmaf(0.353553385f, t, dyl[9]);
          dyl[11] = fmaf(0.456435472f, t, dyl[11]);
        }
        pfma(v12_3, a15.y, d12_54);
        pfma(w12_3, b15.y, d12_54);
        { const float t = vdot(sxu12_3, d12_54);
          dyl[10] = fmaf(0.353553385f, t, dyl[10]);
        }
        DVec ds12 = pmul(ux1, v12_1); pfma(ds12, x1, w12_1);
        pfma(ds12, ux2, v12_2); pfma(ds12, x2, w12_2);
        pfma(ds12, ux3, v12_3); pfma(ds12, x3, w12_3);
        if (gw) gw[12 * NQV] = ds12;
        pfma(dxp[1], us12, v12_1); pfma(dxp[1], s12, w12_1);
        pfma(dxp[2], us12, v12_2); pfma(dxp[2], s12, w12_2);
        pfma(dxp[3], us12, v12_3); pfma(dxp[3], s12, w12_3);
    }
};
}  // namespace
}  // namespace fast

extern const FastKernels kFast_w64_l3;
const FastKernels kFast_w64_l3 = {
    "64|0e+1o|3|0:0:0,1:1:0,0:1:1,1:0:1,1:2:1,1:1:1,0:2:2,1:1:2,1:3:2,1:2:2,0:3:3,1:2:3,1:3:3",
    &fast::fwd_scratch_bytes<fast::Sig_w64_l3>, &fast::bwd_scratch_bytes<fast::Sig_w64_l3>, &fast::launch_fwd<fast::Sig_w64_l3>, &fast::launch_bwd<fast::Sig_w64_l3>, &fast::launch_tp_fwd<fast::Sig_w64_l3>, &fast::launch_tp_bwd<fast::Sig_w64_l3>,
    &fast::launch_dbl_edges<fast::Sig_w64_l3>, &fast::launch_dbl_out<fast::Sig_w64_l3>, nullptr, &fast::launch_bwd_sched<fast::Sig_w64_l3>, 10};
}  // namespace e3j
