// GENERATED by csrc/gen_fast.py from fast/signatures.json -- do not edit.
// signature: 128|0e+1o+2e+3o|2|0:0:0,1:1:0,2:2:0,0:1:1,1:0:1,1:2:1,2:1:1,3:2:1,1:1:1,2:2:1,0:2:2,1:1:2,2:0:2,2:2:2,3:1:2,1:2:2,2:1:2,3:2:2
// 128x0e+128x1o+128x2e+128x3o (x) harmonics l<=2: P=18 D=64 nnz=207 pairs=195
#include "fast_fwd.cuh"
#include "fast_bwd.cuh"
#include "fast_launch.cuh"

namespace e3j {
namespace fast {
namespace {
__device__ const PairRec kPair_q128_l2[200] = {
    {0,1}, {1,1}, {2,1}, {3,1}, {4,1}, {5,1}, {6,1}, {7,1}, {8,1}, {9,1}, {10,1}, {11,1}, {12,1}, {13,1}, {14,1}, {15,2}, {17,1}, {18,1}, {19,1}, {20,1}, {21,1}, {22,1}, {23,1}, {24,2}, {26,1}, {27,1}, {28,1}, {29,1}, {30,1}, {31,1}, {32,1}, {33,1}, {34,1}, {35,1}, {36,1}, {37,0}, {37,1}, {38,1}, {39,2}, {41,1}, {42,1}, {43,1}, {44,1}, {45,1}, {46,1}, {47,1}, {48,1}, {49,1}, {50,1}, {51,1}, {52,1}, {53,1}, {54,2}, {56,1}, {57,1}, {58,1}, {59,1}, {60,1}, {61,1}, {62,1}, {63,1}, {64,1}, {65,1}, {66,1}, {67,2}, {69,1}, {70,1}, {71,1}, {72,1}, {73,1}, {74,1}, {75,2}, {77,1}, {78,1}, {79,1}, {80,1}, {81,1}, {82,1}, {83,1}, {84,1}, {85,1}, {86,1}, {87,1}, {88,1}, {89,1}, {90,1}, {91,1}, {92,0}, {92,1}, {93,1}, {94,1}, {95,1}, {96,1}, {97,1}, {98,1}, {99,1}, {100,1}, {101,1}, {102,1}, {103,1}, {104,1}, {105,1}, {106,2}, {108,1}, {109,1}, {110,1}, {111,1}, {112,1}, {113,1}, {114,1}, {115,1}, {116,1}, {117,1}, {118,1}, {119,2}, {121,1}, {122,1}, {123,1}, {124,1}, {125,1}, {126,1}, {127,1}, {128,1}, {129,1}, {130,1}, {131,1}, {132,1}, {133,1}, {134,1}, {135,1}, {136,1}, {137,1}, {138,1}, {139,1}, {140,1}, {141,1}, {142,1}, {143,1}, {144,1}, {145,1}, {146,1}, {147,0}, {147,0}, {147,0}, {147,1}, {148,1}, {149,1}, {150,1}, {151,1}, {152,2}, {154,1}, {155,1}, {156,2}, {158,1}, {159,1}, {160,1}, {161,1}, {162,1}, {163,1}, {164,1}, {165,1}, {166,1}, {167,1}, {168,1}, {169,1}, {170,1}, {171,1}, {172,1}, {173,1}, {174,1}, {175,1}, {176,1}, {177,1}, {178,1}, {179,1}, {180,1}, {181,1}, {182,1}, {183,1}, {184,1}, {185,1}, {186,1}, {187,1}, {188,2}, {190,1}, {191,1}, {192,1}, {193,1}, {194,1}, {195,1}, {196,2}, {198,1}, {199,1}, {200,1}, {201,1}, {202,1}, {203,1}, {204,1}, {205,1}, {206,1}};
__device__ const float kVal_q128_l2[207] = {
    1.0f, 0.577350259f, 0.577350259f, 0.577350259f, 0.44721359f, 0.44721359f, 0.44721359f, 0.44721359f, 0.44721359f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 0.316227764f, 0.547722578f, -0.547722578f, -0.547722578f, -0.547722578f, -0.632455528f, -0.547722578f, -0.547722578f, -0.547722578f, 0.316227764f, -0.547722578f, 0.547722578f, 0.547722578f, -0.316227764f, -0.547722578f, 0.547722578f, 0.632455528f, 0.547722578f, 0.547722578f, -0.316227764f, 0.547722578f, 0.547722578f, 0.462910056f, 0.377964467f, 0.414039344f, 0.119522862f, -0.292770028f, -0.119522862f, -0.377964467f, -0.462910056f, 0.377964467f, 0.478091449f, 0.507092535f, 0.478091449f, 0.377964467f, 0.462910056f, 0.377964467f, -0.119522862f, -0.292770028f, 0.414039344f, -0.119522862f, 0.377964467f, 0.462910056f, 0.707106769f, -0.707106769f, -0.707106769f, 0.707106769f, 0.707106769f, -0.707106769f, 0.316227764f, -0.316227764f, -0.547722578f, 0.547722578f, -0.316227764f, 0.316227764f, 0.632455528f, 0.316227764f, -0.316227764f, -0.632455528f, -0.316227764f, -0.547722578f, -0.316227764f, 0.547722578f, 0.316227764f, 0.316227764f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 0.707106769f, 0.707106769f, 0.707106769f, 0.707106769f, -0.408248305f, 0.816496611f, -0.408248305f, 0.707106769f, 0.707106769f, -0.707106769f, 0.707106769f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 0.534522474f, -0.462910056f, 0.534522474f, -0.462910056f, -0.462910056f, -0.267261237f, 0.462910056f, -0.267261237f, -0.462910056f, 0.462910056f, 0.534522474f, -0.267261237f, -0.534522474f, -0.267261237f, 0.534522474f, -0.462910056f, -0.462910056f, -0.267261237f, -0.267261237f, -0.462910056f, -0.462910056f, 0.462910056f, 0.534522474f, -0.462910056f, 0.534522474f, 0.597614288f, 0.487950027f, -0.154303357f, -0.154303357f, -0.597614288f, 0.487950027f, 0.617213428f, -0.377964467f, -0.487950027f, 0.534522474f, 0.654653668f, 0.534522474f, 0.487950027f, -0.377964467f, 0.617213428f, 0.487950027f, 0.597614288f, 0.154303357f, -0.154303357f, 0.487950027f, 0.597614288f, 0.408248305f, 0.816496611f, -0.408248305f, -0.408248305f, 0.408248305f, -0.707106769f, -0.408248305f, -0.707106769f, 0.707106769f, 0.707106769f, -0.408248305f, -0.408248305f, 0.408248305f, 0.408248305f, -0.816496611f, 0.408248305f, 0.408248305f, -0.408248305f, 0.816496611f, -0.408248305f, -0.707106769f, 0.408248305f, -0.408248305f, 0.707106769f, -0.707106769f, 0.408248305f, -0.408248305f, 0.707106769f, -0.408248305f, -0.816496611f, 0.408248305f, 0.408248305f, 0.422577113f, 0.327326834f, 0.267261237f, -0.327326834f, 0.597614288f, 0.422577113f, -0.422577113f, -0.327326834f, -0.534522474f, 0.377964467f, -0.327326834f, -0.422577113f, 0.597614288f, 0.377964467f, -0.377964467f, -0.597614288f, 0.422577113f, -0.377964467f, -0.327326834f, 0.534522474f, 0.327326834f, -0.422577113f, -0.422577113f, -0.597614288f, 0.327326834f, -0.267261237f, 0.327326834f, 0.422577113f};
__device__ const unsigned char kI2_q128_l2[207] = {
    0, 1, 2, 3, 4, 5, 6, 7, 8, 1, 2, 3, 0, 0, 0, 6, 8, 5, 4, 5, 6, 7, 4, 7, 6, 8, 3, 2, 1, 1, 1, 2, 3, 1, 3, 2, 3, 8, 7, 6, 8, 5, 4, 5, 4, 4, 5, 6, 7, 8, 4, 5, 4, 7, 6, 8, 7, 8, 3, 2, 3, 1, 2, 1, 5, 4, 7, 6, 8, 7, 8, 7, 5, 4, 7, 6, 8, 5, 4, 5, 4, 5, 6, 7, 8, 3, 1, 2, 1, 1, 2, 3, 3, 2, 1, 3, 0, 0, 0, 0, 0, 6, 7, 4, 5, 7, 6, 8, 5, 4, 5, 4, 5, 6, 7, 8, 5, 4, 7, 6, 8, 7, 5, 8, 7, 6, 3, 2, 3, 1, 1, 3, 2, 1, 1, 1, 2, 3, 1, 3, 2, 3, 1, 1, 3, 2, 3, 5, 8, 7, 4, 7, 6, 8, 7, 5, 6, 8, 5, 4, 7, 4, 5, 1, 3, 2, 1, 3, 2, 3, 3, 1, 3, 2, 1, 1, 2, 3, 1, 5, 5, 8, 7, 6, 7, 4, 4, 7, 6, 8, 8, 8, 7, 5, 4, 8, 6, 8, 5, 4, 4, 7, 6, 7, 4, 5, 5};
__device__ const PairRec kBPair_q128_l2[204] = {
    {0,1}, {1,1}, {2,1}, {3,1}, {4,1}, {5,1}, {6,1}, {7,1}, {8,1}, {9,1}, {10,1}, {11,1}, {12,1}, {13,1}, {14,1}, {15,1}, {16,1}, {17,1}, {18,1}, {19,1}, {20,1}, {21,1}, {22,1}, {23,1}, {24,1}, {25,1}, {26,1}, {27,1}, {28,1}, {29,1}, {30,1}, {31,1}, {32,2}, {34,1}, {35,1}, {36,1}, {37,1}, {38,1}, {39,1}, {40,2}, {42,1}, {43,1}, {44,1}, {45,1}, {46,1}, {47,1}, {48,1}, {49,1}, {50,1}, {51,0}, {51,0}, {51,0}, {51,1}, {52,1}, {53,1}, {54,1}, {55,1}, {56,1}, {57,2}, {59,1}, {60,1}, {61,1}, {62,1}, {63,1}, {64,1}, {65,1}, {66,2}, {68,1}, {69,1}, {70,1}, {71,1}, {72,1}, {73,1}, {74,1}, {75,1}, {76,1}, {77,1}, {78,1}, {79,1}, {80,1}, {81,1}, {82,1}, {83,1}, {84,1}, {85,1}, {86,1}, {87,1}, {88,1}, {89,1}, {90,1}, {91,1}, {92,1}, {93,1}, {94,2}, {96,1}, {97,1}, {98,2}, {100,1}, {101,1}, {102,1}, {103,1}, {104,1}, {105,0}, {105,0}, {105,1}, {106,1}, {107,1}, {108,1}, {109,1}, {110,1}, {111,1}, {112,2}, {114,1}, {115,1}, {116,1}, {117,1}, {118,1}, {119,1}, {120,1}, {121,1}, {122,1}, {123,1}, {124,1}, {125,1}, {126,1}, {127,2}, {129,1}, {130,1}, {131,1}, {132,1}, {133,1}, {134,1}, {135,1}, {136,1}, {137,1}, {138,1}, {139,1}, {140,1}, {141,1}, {142,1}, {143,1}, {144,1}, {145,1}, {146,1}, {147,1}, {148,1}, {149,1}, {150,1}, {151,1}, {152,0}, {152,0}, {152,0}, {152,1}, {153,1}, {154,1}, {155,1}, {156,1}, {157,1}, {158,2}, {160,1}, {161,1}, {162,1}, {163,1}, {164,1}, {165,1}, {166,2}, {168,1}, {169,1}, {170,1}, {171,1}, {172,1}, {173,1}, {174,1}, {175,1}, {176,1}, {177,1}, {178,1}, {179,1}, {180,1}, {181,1}, {182,1}, {183,1}, {184,1}, {185,1}, {186,1}, {187,2}, {189,1}, {190,1}, {191,1}, {192,1}, {193,1}, {194,1}, {195,1}, {196,1}, {197,1}, {198,1}, {199,1}, {200,2}, {202,1}, {203,1}, {204,1}, {205,1}, {206,1}, {207,0}};
__device__ const float kBVal_q128_l2[207] = {
    1.0f, 0.547722578f, 0.547722578f, -0.316227764f, -0.547722578f, 0.547722578f, 0.632455528f, 0.547722578f, 0.547722578f, -0.316227764f, 0.547722578f, 0.547722578f, 0.707106769f, -0.707106769f, -0.707106769f, 0.707106769f, 0.707106769f, -0.707106769f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 0.422577113f, 0.327326834f, 0.267261237f, -0.327326834f, 0.597614288f, 0.422577113f, -0.422577113f, -0.327326834f, -0.534522474f, 0.377964467f, -0.327326834f, -0.422577113f, 0.597614288f, 0.377964467f, -0.377964467f, -0.597614288f, 0.422577113f, -0.377964467f, -0.327326834f, 0.534522474f, 0.327326834f, -0.422577113f, -0.422577113f, -0.597614288f, 0.327326834f, -0.267261237f, 0.327326834f, 0.422577113f, 0.577350259f, 0.577350259f, 0.577350259f, 1.0f, 1.0f, 1.0f, 0.316227764f, 0.547722578f, -0.547722578f, -0.547722578f, -0.547722578f, -0.632455528f, -0.547722578f, -0.547722578f, -0.547722578f, 0.316227764f, -0.547722578f, 0.597614288f, 0.487950027f, -0.154303357f, -0.154303357f, -0.597614288f, 0.487950027f, 0.617213428f, -0.377964467f, -0.487950027f, 0.534522474f, 0.654653668f, 0.534522474f, 0.487950027f, -0.377964467f, 0.617213428f, 0.487950027f, 0.597614288f, 0.154303357f, -0.154303357f, 0.487950027f, 0.597614288f, 0.408248305f, 0.816496611f, -0.408248305f, -0.408248305f, 0.408248305f, -0.707106769f, -0.408248305f, -0.707106769f, 0.707106769f, 0.707106769f, -0.408248305f, -0.408248305f, 0.408248305f, 0.408248305f, -0.816496611f, 0.408248305f, 0.44721359f, 0.44721359f, 0.44721359f, 0.44721359f, 0.44721359f, 0.462910056f, 0.377964467f, 0.414039344f, 0.119522862f, -0.292770028f, -0.119522862f, -0.377964467f, -0.462910056f, 0.377964467f, 0.478091449f, 0.507092535f, 0.478091449f, 0.377964467f, 0.462910056f, 0.377964467f, -0.119522862f, -0.292770028f, 0.414039344f, -0.119522862f, 0.377964467f, 0.462910056f, 1.0f, 1.0f, 1.0f, 1.0f, 1.0f, 0.408248305f, -0.408248305f, 0.816496611f, -0.408248305f, -0.707106769f, 0.408248305f, -0.408248305f, 0.707106769f, -0.707106769f, 0.408248305f, -0.408248305f, 0.707106769f, -0.408248305f, -0.816496611f, 0.408248305f, 0.408248305f, 1.0f, 1.0f, 1.0f, 0.316227764f, -0.316227764f, -0.547722578f, 0.547722578f, -0.316227764f, 0.316227764f, 0.632455528f, 0.316227764f, -0.316227764f, -0.632455528f, -0.316227764f, -0.547722578f, -0.316227764f, 0.547722578f, 0.316227764f, 0.316227764f, 0.707106769f, 0.707106769f, 0.707106769f, 0.707106769f, -0.408248305f, 0.816496611f, -0.408248305f, 0.707106769f, 0.707106769f, -0.707106769f, 0.707106769f, 0.534522474f, -0.462910056f, 0.534522474f, -0.462910056f, -0.462910056f, -0.267261237f, 0.462910056f, -0.267261237f, -0.462910056f, 0.462910056f, 0.534522474f, -0.267261237f, -0.534522474f, -0.267261237f, 0.534522474f, -0.462910056f, -0.462910056f, -0.267261237f, -0.267261237f, -0.462910056f, -0.462910056f, 0.462910056f, 0.534522474f, -0.462910056f, 0.534522474f};
__device__ const unsigned char kBI2_q128_l2[207] = {
    0, 3, 2, 1, 1, 1, 2, 3, 1, 3, 2, 3, 3, 2, 3, 1, 2, 1, 4, 5, 6, 7, 8, 5, 5, 8, 7, 6, 7, 4, 4, 7, 6, 8, 8, 8, 7, 5, 4, 8, 6, 8, 5, 4, 4, 7, 6, 7, 4, 5, 5, 1, 2, 3, 1, 2, 3, 6, 8, 5, 4, 5, 6, 7, 4, 7, 6, 8, 3, 2, 3, 1, 1, 3, 2, 1, 1, 1, 2, 3, 1, 3, 2, 3, 1, 1, 3, 2, 3, 5, 8, 7, 4, 7, 6, 8, 7, 5, 6, 8, 5, 4, 7, 4, 5, 4, 5, 6, 7, 8, 8, 7, 6, 8, 5, 4, 5, 4, 4, 5, 6, 7, 8, 4, 5, 4, 7, 6, 8, 7, 8, 0, 0, 0, 0, 0, 1, 3, 2, 1, 3, 2, 3, 3, 1, 3, 2, 1, 1, 2, 3, 1, 0, 0, 0, 5, 4, 7, 6, 8, 7, 8, 7, 5, 4, 7, 6, 8, 5, 4, 5, 3, 1, 2, 1, 1, 2, 3, 3, 2, 1, 3, 6, 7, 4, 5, 7, 6, 8, 5, 4, 5, 4, 5, 6, 7, 8, 5, 4, 7, 6, 8, 7, 5, 8, 7, 6};
__device__ const unsigned char kBRow_q128_l2[68] = {
    0, 12, 13, 14, 18, 19, 20, 24, 25, 26, 27, 28, 59, 60, 61, 62, 63, 1, 3, 4, 5, 9, 10, 11, 44, 45, 46, 47, 48, 49, 50, 51, 52, 53, 2, 15, 16, 17, 34, 35, 36, 37, 38, 54, 55, 56, 57, 58, 58, 58, 58, 6, 7, 8, 21, 22, 23, 29, 30, 31, 32, 33, 39, 40, 41, 42, 43, 43};

struct Sig_q128_l2 {
    static constexpr int NQ = 128, DIN = 16, DSH = 9, P = 18, D = 64;
    static constexpr int NNZ = 207, NPAIR = 195, V = 4;
    static constexpr int FW = 4, FT = 3, FS = 2, FC = 2, F_RMAX = 17, F_APAD = 200, F_NREC = 2, F_NPMAX = 56, F_MAXREG = 255;
    // fused double backward (cotangent of grad_out): tile, stages, CTAs per SM (DFT = 0: not generated)
    static constexpr int DFT = 0, DFS = 2, DFC = 1, DFV = 4;
    using DFVec = float4;
    using Vec = float4;
    __device__ static __forceinline__ PairRec pair_rec(int i) { return kPair_q128_l2[i]; }
    __device__ static __forceinline__ float rec_val(int i) { return kVal_q128_l2[i]; }
    __device__ static __forceinline__ unsigned char rec_i2(int i) { return kI2_q128_l2[i]; }
    static constexpr int f_row0(int g) {
        switch (g) {
            case 0: return 0;
            case 1: return 15;
            case 2: return 32;
            case 3: return 49;
            case 4: return 64;
            default: return 64;
        }
    }
    static constexpr int f_a0(int g) {
        switch (g) {
            case 0: return 0;
            case 1: return 36;
            case 2: return 88;
            case 3: return 144;
            case 4: return 200;
            default: return 200;
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
            const Vec x4 = xs[4 * NQV];
            const Vec x5 = xs[5 * NQV];
            const Vec x6 = xs[6 * NQV];
            const Vec x7 = xs[7 * NQV];
            const Vec x8 = xs[8 * NQV];
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
            const Vec s2 = ss[2 * NQV];  // path 2: l1=2 l2=2 -> L=0
            const Vec sx2_4 = pmul(s2, x4);
            const Vec sx2_5 = pmul(s2, x5);
            const Vec sx2_6 = pmul(s2, x6);
            const Vec sx2_7 = pmul(s2, x7);
            const Vec sx2_8 = pmul(s2, x8);
            const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
            pfma(acc[2], a1.x, sx2_4);
            pfma(acc[2], a1.y, sx2_5);
            pfma(acc[2], a1.z, sx2_6);
            pfma(acc[2], a1.w, sx2_7);
            const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
            pfma(acc[2], a2.x, sx2_8);
            const Vec s3 = ss[3 * NQV];  // path 3: l1=0 l2=1 -> L=1
            const Vec sx3_0 = pmul(s3, x0);
            pfma(acc[3], a2.y, sx3_0);
            pfma(acc[4], a2.z, sx3_0);
            pfma(acc[5], a2.w, sx3_0);
            const Vec s4 = ss[4 * NQV];  // path 4: l1=1 l2=0 -> L=1
            const Vec sx4_1 = pmul(s4, x1);
            const Vec sx4_2 = pmul(s4, x2);
            const Vec sx4_3 = pmul(s4, x3);
            const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
            pfma(acc[6], a3.x, sx4_1);
            pfma(acc[7], a3.y, sx4_2);
            pfma(acc[8], a3.z, sx4_3);
            const Vec s5 = ss[5 * NQV];  // path 5: l1=1 l2=2 -> L=1
            const Vec sx5_1 = pmul(s5, x1);
            const Vec sx5_2 = pmul(s5, x2);
            const Vec sx5_3 = pmul(s5, x3);
            pfma(acc[9], a3.w, sx5_1);
            const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
            pfma(acc[10], a4.z, sx5_1);
            const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
            pfma(acc[11], a5.y, sx5_1);
            pfma(acc[9], a4.x, sx5_2);
            pfma(acc[10], a4.w, sx5_2);
            pfma(acc[11], a5.z, sx5_2);
            pfma(acc[9], a4.y, sx5_3);
            pfma(acc[10], a5.x, sx5_3);
            pfma(acc[11], a5.w, sx5_3);
            const Vec s6 = ss[6 * NQV];  // path 6: l1=2 l2=1 -> L=1
            const Vec sx6_4 = pmul(s6, x4);
            const Vec sx6_5 = pmul(s6, x5);
            const Vec sx6_6 = pmul(s6, x6);
            const Vec sx6_7 = pmul(s6, x7);
            const Vec sx6_8 = pmul(s6, x8);
            const float4 a6 = *reinterpret_cast<const float4*>(As + 24);
            pfma(acc[12], a6.x, sx6_4);
            const float4 a7 = *reinterpret_cast<const float4*>(As + 28);
            pfma(acc[13], a7.x, sx6_5);
            pfma(acc[14], a7.w, sx6_4);
            pfma(acc[12], a6.y, sx6_5);
            pfma(acc[13], a7.y, sx6_6);
            const float4 a8 = *reinterpret_cast<const float4*>(As + 32);
            pfma(acc[14], a8.x, sx6_6);
            pfma(acc[12], a6.z, sx6_6);
            pfma(acc[13], a7.z, sx6_7);
            pfma(acc[14], a8.y, sx6_7);
            pfma(acc[12], a6.w, sx6_8);
            pfma(acc[14], a8.z, sx6_8);
        }
        if constexpr (G == 1) {
            const Vec x0 = xs[0 * NQV];
            const Vec x1 = xs[1 * NQV];
            const Vec x2 = xs[2 * NQV];
            const Vec x3 = xs[3 * NQV];
            const Vec x4 = xs[4 * NQV];
            const Vec x5 = xs[5 * NQV];
            const Vec x6 = xs[6 * NQV];
            const Vec x7 = xs[7 * NQV];
            const Vec x8 = xs[8 * NQV];
            const Vec x9 = xs[9 * NQV];
            const Vec x10 = xs[10 * NQV];
            const Vec x11 = xs[11 * NQV];
            const Vec x12 = xs[12 * NQV];
            const Vec x13 = xs[13 * NQV];
            const Vec x14 = xs[14 * NQV];
            const Vec x15 = xs[15 * NQV];
            const Vec s7 = ss[7 * NQV];  // path 7: l1=3 l2=2 -> L=1
            const Vec sx7_9 = pmul(s7, x9);
            const Vec sx7_10 = pmul(s7, x10);
            const Vec sx7_11 = pmul(s7, x11);
            const Vec sx7_12 = pmul(s7, x12);
            const Vec sx7_13 = pmul(s7, x13);
            const Vec sx7_14 = pmul(s7, x14);
            const Vec sx7_15 = pmul(s7, x15);
            const float4 a9 = *reinterpret_cast<const float4*>(As + 36);
            pfma(acc[0], a9.x, sx7_9);
            const float4 a10 = *reinterpret_cast<const float4*>(As + 40);
            pfma(acc[1], a10.w, sx7_10);
            const float4 a12 = *reinterpret_cast<const float4*>(As + 48);
            pfma(acc[2], a12.x, sx7_9);
            pfma(acc[0], a9.y, sx7_10);
            const float4 a11 = *reinterpret_cast<const float4*>(As + 44);
            pfma(acc[1], a11.x, sx7_11);
            pfma(acc[2], a12.y, sx7_10);
            pfma(acc[0], a9.z, sx7_11);
            pfma(acc[1], a11.y, sx7_12);
            pfma(acc[2], a12.z, sx7_11);
            pfma(acc[0], a9.w, sx7_12);
            pfma(acc[1], a11.z, sx7_13);
            pfma(acc[2], a12.w, sx7_12);
            pfma(acc[0], a10.x, sx7_13);
            pfma(acc[1], a11.w, sx7_14);
            const float4 a13 = *reinterpret_cast<const float4*>(As + 52);
            pfma(acc[2], a13.x, sx7_13);
            pfma(acc[0], a10.y, sx7_14);
            pfma(acc[2], a13.y, sx7_14);
            pfma(acc[0], a10.z, sx7_15);
            pfma(acc[2], a13.z, sx7_15);
            const Vec s8 = ss[8 * NQV];  // path 8: l1=1 l2=1 -> L=1
            const Vec sx8_1 = pmul(s8, x1);
            const Vec sx8_2 = pmul(s8, x2);
            const Vec sx8_3 = pmul(s8, x3);
            pfma(acc[3], a13.w, sx8_2);
            const float4 a14 = *reinterpret_cast<const float4*>(As + 56);
            pfma(acc[4], a14.y, sx8_1);
            pfma(acc[5], a14.w, sx8_1);
            pfma(acc[3], a14.x, sx8_3);
            pfma(acc[4], a14.z, sx8_3);
            const float4 a15 = *reinterpret_cast<const float4*>(As + 60);
            pfma(acc[5], a15.x, sx8_2);
            const Vec s9 = ss[9 * NQV];  // path 9: l1=2 l2=2 -> L=1
            const Vec sx9_4 = pmul(s9, x4);
            const Vec sx9_5 = pmul(s9, x5);
            const Vec sx9_6 = pmul(s9, x6);
            const Vec sx9_7 = pmul(s9, x7);
            const Vec sx9_8 = pmul(s9, x8);
            pfma(acc[6], a15.y, sx9_4);
            const float4 a16 = *reinterpret_cast<const float4*>(As + 64);
            pfma(acc[7], a16.z, sx9_4);
            const float4 a17 = *reinterpret_cast<const float4*>(As + 68);
            pfma(acc[8], a17.z, sx9_4);
            pfma(acc[6], a15.z, sx9_5);
            pfma(acc[7], a16.w, sx9_5);
            pfma(acc[8], a17.w, sx9_5);
            pfma(acc[6], a15.w, sx9_6);
            pfma(acc[7], a17.x, sx9_7);
            const float4 a18 = *reinterpret_cast<const float4*>(As + 72);
            pfma(acc[8], a18.x, sx9_6);
            pfma(acc[6], a16.x, sx9_7);
            pfma(acc[7], a17.y, sx9_8);
            pfma(acc[8], a18.y, sx9_7);
            pfma(acc[6], a16.y, sx9_8);
            pfma(acc[8], a18.z, sx9_8);
            const Vec s10 = ss[10 * NQV];  // path 10: l1=0 l2=2 -> L=2
            const Vec sx10_0 = pmul(s10, x0);
            pfma(acc[9], a18.w, sx10_0);
            const float4 a19 = *reinterpret_cast<const float4*>(As + 76);
            pfma(acc[10], a19.x, sx10_0);
            pfma(acc[11], a19.y, sx10_0);
            pfma(acc[12], a19.z, sx10_0);
            pfma(acc[13], a19.w, sx10_0);
            const Vec s11 = ss[11 * NQV];  // path 11: l1=1 l2=1 -> L=2
            const Vec sx11_1 = pmul(s11, x1);
            const Vec sx11_2 = pmul(s11, x2);
            const Vec sx11_3 = pmul(s11, x3);
            const float4 a20 = *reinterpret_cast<const float4*>(As + 80);
            pfma(acc[14], a20.x, sx11_1);
            pfma(acc[15], a20.z, sx11_1);
            const float4 a21 = *reinterpret_cast<const float4*>(As + 84);
            pfma(acc[16], a21.x, sx11_1);
            pfma(acc[14], a20.y, sx11_3);
            pfma(acc[15], a20.w, sx11_2);
            pfma(acc[16], a21.y, sx11_2);
            pfma(acc[16], a21.z, sx11_3);
        }
        if constexpr (G == 2) {
            const Vec x1 = xs[1 * NQV];
            const Vec x2 = xs[2 * NQV];
            const Vec x3 = xs[3 * NQV];
            const Vec x4 = xs[4 * NQV];
            const Vec x5 = xs[5 * NQV];
            const Vec x6 = xs[6 * NQV];
            const Vec x7 = xs[7 * NQV];
            const Vec x8 = xs[8 * NQV];
            const Vec x9 = xs[9 * NQV];
            const Vec x10 = xs[10 * NQV];
            const Vec x11 = xs[11 * NQV];
            const Vec x12 = xs[12 * NQV];
            const Vec x13 = xs[13 * NQV];
            const Vec x14 = xs[14 * NQV];
            const Vec x15 = xs[15 * NQV];
            const Vec s11 = ss[11 * NQV];  // path 11: l1=1 l2=1 -> L=2
            const Vec sx11_1 = pmul(s11, x1);
            const Vec sx11_2 = pmul(s11, x2);
            const Vec sx11_3 = pmul(s11, x3);
            const float4 a22 = *reinterpret_cast<const float4*>(As + 88);
            pfma(acc[0], a22.x, sx11_2);
            pfma(acc[1], a22.z, sx11_1);
            pfma(acc[0], a22.y, sx11_3);
            pfma(acc[1], a22.w, sx11_3);
            const Vec s12 = ss[12 * NQV];  // path 12: l1=2 l2=0 -> L=2
            const Vec sx12_4 = pmul(s12, x4);
            const Vec sx12_5 = pmul(s12, x5);
            const Vec sx12_6 = pmul(s12, x6);
            const Vec sx12_7 = pmul(s12, x7);
            const Vec sx12_8 = pmul(s12, x8);
            const float4 a23 = *reinterpret_cast<const float4*>(As + 92);
            pfma(acc[2], a23.x, sx12_4);
            pfma(acc[3], a23.y, sx12_5);
            pfma(acc[4], a23.z, sx12_6);
            pfma(acc[5], a23.w, sx12_7);
            const float4 a24 = *reinterpret_cast<const float4*>(As + 96);
            pfma(acc[6], a24.x, sx12_8);
            const Vec s13 = ss[13 * NQV];  // path 13: l1=2 l2=2 -> L=2
            const Vec sx13_4 = pmul(s13, x4);
            const Vec sx13_5 = pmul(s13, x5);
            const Vec sx13_6 = pmul(s13, x6);
            const Vec sx13_7 = pmul(s13, x7);
            const Vec sx13_8 = pmul(s13, x8);
            pfma(acc[7], a24.y, sx13_4);
            const float4 a25 = *reinterpret_cast<const float4*>(As + 100);
            pfma(acc[8], a25.y, sx13_4);
            const float4 a26 = *reinterpret_cast<const float4*>(As + 104);
            pfma(acc[9], a26.z, sx13_4);
            const float4 a27 = *reinterpret_cast<const float4*>(As + 108);
            pfma(acc[10], a27.w, sx13_4);
            const float4 a29 = *reinterpret_cast<const float4*>(As + 116);
            pfma(acc[11], a29.x, sx13_5);
            pfma(acc[7], a24.z, sx13_5);
            pfma(acc[8], a25.z, sx13_5);
            pfma(acc[9], a26.w, sx13_5);
            const float4 a28 = *reinterpret_cast<const float4*>(As + 112);
            pfma(acc[10], a28.x, sx13_5);
            pfma(acc[11], a29.y, sx13_6);
            pfma(acc[7], a24.w, sx13_6);
            pfma(acc[8], a25.w, sx13_6);
            pfma(acc[9], a27.x, sx13_6);
            pfma(acc[10], a28.y, sx13_6);
            pfma(acc[11], a29.z, sx13_7);
            pfma(acc[7], a25.x, sx13_7);
            pfma(acc[8], a26.x, sx13_7);
            pfma(acc[9], a27.y, sx13_7);
            pfma(acc[10], a28.z, sx13_7);
            pfma(acc[11], a29.w, sx13_8);
            pfma(acc[8], a26.y, sx13_8);
            pfma(acc[9], a27.z, sx13_8);
            pfma(acc[10], a28.w, sx13_8);
            const Vec s14 = ss[14 * NQV];  // path 14: l1=3 l2=1 -> L=2
            const Vec sx14_9 = pmul(s14, x9);
            const Vec sx14_10 = pmul(s14, x10);
            const Vec sx14_11 = pmul(s14, x11);
            const Vec sx14_12 = pmul(s14, x12);
            const Vec sx14_13 = pmul(s14, x13);
            const Vec sx14_14 = pmul(s14, x14);
            const Vec sx14_15 = pmul(s14, x15);
            const float4 a30 = *reinterpret_cast<const float4*>(As + 120);
            pfma(acc[12], a30.x, sx14_9);
            const float4 a31 = *reinterpret_cast<const float4*>(As + 124);
            pfma(acc[13], a31.y, sx14_10);
            const float4 a32 = *reinterpret_cast<const float4*>(As + 128);
            pfma(acc[14], a32.y, sx14_11);
            const float4 a33 = *reinterpret_cast<const float4*>(As + 132);
            pfma(acc[15], a33.x, sx14_10);
            const float4 a34 = *reinterpret_cast<const float4*>(As + 136);
            pfma(acc[16], a34.x, sx14_9);
            pfma(acc[12], a30.y, sx14_10);
            pfma(acc[13], a31.z, sx14_11);
            pfma(acc[14], a32.z, sx14_12);
            pfma(acc[15], a33.y, sx14_12);
            pfma(acc[16], a34.y, sx14_11);
            pfma(acc[12], a30.z, sx14_11);
            pfma(acc[13], a31.w, sx14_12);
            pfma(acc[14], a32.w, sx14_13);
            pfma(acc[15], a33.z, sx14_13);
            pfma(acc[16], a34.z, sx14_13);
            pfma(acc[12], a30.w, sx14_13);
            pfma(acc[13], a32.x, sx14_14);
            pfma(acc[15], a33.w, sx14_14);
            pfma(acc[16], a34.w, sx14_14);
            pfma(acc[12], a31.x, sx14_15);
            const float4 a35 = *reinterpret_cast<const float4*>(As + 140);
            pfma(acc[16], a35.x, sx14_15);
        }
        if constexpr (G == 3) {
            const Vec x1 = xs[1 * NQV];
            const Vec x2 = xs[2 * NQV];
            const Vec x3 = xs[3 * NQV];
            const Vec x4 = xs[4 * NQV];
            const Vec x5 = xs[5 * NQV];
            const Vec x6 = xs[6 * NQV];
            const Vec x7 = xs[7 * NQV];
            const Vec x8 = xs[8 * NQV];
            const Vec x9 = xs[9 * NQV];
            const Vec x10 = xs[10 * NQV];
            const Vec x11 = xs[11 * NQV];
            const Vec x12 = xs[12 * NQV];
            const Vec x13 = xs[13 * NQV];
            const Vec x14 = xs[14 * NQV];
            const Vec x15 = xs[15 * NQV];
            const Vec s15 = ss[15 * NQV];  // path 15: l1=1 l2=2 -> L=2
            const Vec sx15_1 = pmul(s15, x1);
            const Vec sx15_2 = pmul(s15, x2);
            const Vec sx15_3 = pmul(s15, x3);
            const float4 a36 = *reinterpret_cast<const float4*>(As + 144);
            pfma(acc[0], a36.x, sx15_1);
            pfma(acc[1], a36.w, sx15_1);
            const float4 a37 = *reinterpret_cast<const float4*>(As + 148);
            pfma(acc[2], a37.z, sx15_1);
            const float4 a38 = *reinterpret_cast<const float4*>(As + 152);
            pfma(acc[3], a38.x, sx15_1);
            pfma(acc[4], a38.w, sx15_1);
            pfma(acc[0], a36.y, sx15_2);
            pfma(acc[1], a37.x, sx15_2);
            pfma(acc[2], a37.w, sx15_3);
            pfma(acc[3], a38.y, sx15_2);
            const float4 a39 = *reinterpret_cast<const float4*>(As + 156);
            pfma(acc[4], a39.x, sx15_2);
            pfma(acc[0], a36.z, sx15_3);
            pfma(acc[1], a37.y, sx15_3);
            pfma(acc[3], a38.z, sx15_3);
            pfma(acc[4], a39.y, sx15_3);
            const Vec s16 = ss[16 * NQV];  // path 16: l1=2 l2=1 -> L=2
            const Vec sx16_4 = pmul(s16, x4);
            const Vec sx16_5 = pmul(s16, x5);
            const Vec sx16_6 = pmul(s16, x6);
            const Vec sx16_7 = pmul(s16, x7);
            const Vec sx16_8 = pmul(s16, x8);
            pfma(acc[5], a39.z, sx16_5);
            const float4 a40 = *reinterpret_cast<const float4*>(As + 160);
            pfma(acc[6], a40.y, sx16_4);
            const float4 a41 = *reinterpret_cast<const float4*>(As + 164);
            pfma(acc[7], a41.y, sx16_5);
            pfma(acc[8], a41.w, sx16_4);
            const float4 a42 = *reinterpret_cast<const float4*>(As + 168);
            pfma(acc[9], a42.w, sx16_4);
            pfma(acc[5], a39.w, sx16_7);
            pfma(acc[6], a40.z, sx16_6);
            pfma(acc[7], a41.z, sx16_7);
            pfma(acc[8], a42.x, sx16_5);
            const float4 a43 = *reinterpret_cast<const float4*>(As + 172);
            pfma(acc[9], a43.x, sx16_5);
            pfma(acc[5], a40.x, sx16_8);
            pfma(acc[6], a40.w, sx16_7);
            pfma(acc[8], a42.y, sx16_6);
            pfma(acc[9], a43.y, sx16_7);
            pfma(acc[6], a41.x, sx16_8);
            pfma(acc[8], a42.z, sx16_8);
            const Vec s17 = ss[17 * NQV];  // path 17: l1=3 l2=2 -> L=2
            const Vec sx17_9 = pmul(s17, x9);
            const Vec sx17_10 = pmul(s17, x10);
            const Vec sx17_11 = pmul(s17, x11);
            const Vec sx17_12 = pmul(s17, x12);
            const Vec sx17_13 = pmul(s17, x13);
            const Vec sx17_14 = pmul(s17, x14);
            const Vec sx17_15 = pmul(s17, x15);
            pfma(acc[10], a43.z, sx17_9);
            const float4 a45 = *reinterpret_cast<const float4*>(As + 180);
            pfma(acc[11], a45.x, sx17_9);
            const float4 a46 = *reinterpret_cast<const float4*>(As + 184);
            pfma(acc[12], a46.y, sx17_10);
            const float4 a47 = *reinterpret_cast<const float4*>(As + 188);
            pfma(acc[13], a47.y, sx17_9);
            const float4 a48 = *reinterpret_cast<const float4*>(As + 192);
            pfma(acc[14], a48.z, sx17_9);
            pfma(acc[10], a43.w, sx17_11);
            pfma(acc[11], a45.y, sx17_11);
            pfma(acc[12], a46.z, sx17_11);
            pfma(acc[13], a47.z, sx17_11);
            pfma(acc[14], a48.w, sx17_10);
            const float4 a44 = *reinterpret_cast<const float4*>(As + 176);
            pfma(acc[10], a44.x, sx17_12);
            pfma(acc[11], a45.z, sx17_12);
            pfma(acc[12], a46.w, sx17_13);
            pfma(acc[13], a47.w, sx17_12);
            const float4 a49 = *reinterpret_cast<const float4*>(As + 196);
            pfma(acc[14], a49.x, sx17_11);
            pfma(acc[10], a44.y, sx17_13);
            pfma(acc[11], a45.w, sx17_13);
            pfma(acc[12], a47.x, sx17_14);
            pfma(acc[13], a48.x, sx17_13);
            pfma(acc[14], a49.y, sx17_12);
            pfma(acc[10], a44.z, sx17_14);
            pfma(acc[11], a46.x, sx17_15);
            pfma(acc[13], a48.y, sx17_15);
            pfma(acc[14], a49.z, sx17_13);
            pfma(acc[10], a44.w, sx17_15);
            pfma(acc[14], a49.w, sx17_15);
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
            dst[13 * stride] = acc[13];
            dst[14 * stride] = acc[14];
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
            dst[11 * stride] = acc[11];
            dst[12 * stride] = acc[12];
            dst[13 * stride] = acc[13];
            dst[14 * stride] = acc[14];
            dst[15 * stride] = acc[15];
            dst[16 * stride] = acc[16];
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
            dst[16 * stride] = acc[16];
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
    // ---- backward: path groups [[0, 6, 8, 10, 17], [1, 3, 5, 14, 15], [2, 7, 12, 16], [4, 9, 11, 13]]
    static constexpr int BV = 4;  // channels per lane in the backward
    using BVec = float4;
    static constexpr int BW = 4, BT = 4, BS = 2, BC = 1, B_RMAX = 17, B_APAD = 204, B_NREC = 2;
    // edge-wise backward (one warp per edge, grad_out rows read from shared memory): edges per tile (0 = not generated), ring stages
    static constexpr int ET = 4, ES = 2, EV = 2, EXG = 0;   // EXG: sender rows not staged
    static constexpr int ST = 4;   // columns of the scheduled backward
    // the same for the standalone tensor product: rows per ring slot (0 = not generated), ring slots
    static constexpr int ETR = 0, ESR = 3;
    // fused double backward (edge outputs): edges per tile (0 = not generated), ring stages
    static constexpr int DT = 0, DS = 2, DV = 2;
    using DVec = float2;
    using EVec = float2;
    __device__ static __forceinline__ PairRec b_pair_rec(int i) { return kBPair_q128_l2[i]; }
    __device__ static __forceinline__ float b_rec_val(int i) { return kBVal_q128_l2[i]; }
    __device__ static __forceinline__ unsigned char b_rec_i2(int i) { return kBI2_q128_l2[i]; }
    // output rows of path group g: b_nrow(g) of them, the r-th is b_row(g, r)
    __device__ static __forceinline__ int b_row(int g, int r) { return kBRow_q128_l2[g * B_RMAX + r]; }
    static constexpr int b_nrow(int g) {
        switch (g) {
            case 0: return 17;
            case 1: return 17;
            case 2: return 14;
            case 3: return 16;
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
            const BVec x4 = xs[4 * NQV];
            const BVec x5 = xs[5 * NQV];
            const BVec x6 = xs[6 * NQV];
            const BVec x7 = xs[7 * NQV];
            const BVec x8 = xs[8 * NQV];
            const BVec x9 = xs[9 * NQV];
            const BVec x10 = xs[10 * NQV];
            const BVec x11 = xs[11 * NQV];
            const BVec x12 = xs[12 * NQV];
            const BVec x13 = xs[13 * NQV];
            const BVec x14 = xs[14 * NQV];
            const BVec x15 = xs[15 * NQV];
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
            const BVec s6 = ss[6 * NQV];  // path 6: l1=2 l2=1 -> L=1
            const BVec sx6_4 = vmul(s6, x4);
            BVec u6_4; vzero(u6_4);
            const BVec sx6_5 = vmul(s6, x5);
            BVec u6_5; vzero(u6_5);
            const BVec sx6_6 = vmul(s6, x6);
            BVec u6_6; vzero(u6_6);
            const BVec sx6_7 = vmul(s6, x7);
            BVec u6_7; vzero(u6_7);
            const BVec sx6_8 = vmul(s6, x8);
            BVec u6_8; vzero(u6_8);
            vfma(u6_4, a0.y, dm[1]);
            { const float t = vdot(sx6_4, dm[1]);
              dyl[3] = 0.547722578f * t;
            }
            const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
            vfma(u6_5, a1.y, dm[2]);
            { const float t = vdot(sx6_5, dm[2]);
              dyl[1] = 0.547722578f * t;
            }
            const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
            vfma(u6_4, a2.x, dm[3]);
            { const float t = vdot(sx6_4, dm[3]);
              dyl[1] = fmaf(0.547722578f, t, dyl[1]);
            }
            vfma(u6_5, a0.z, dm[1]);
            { const float t = vdot(sx6_5, dm[1]);
              dyl[2] = 0.547722578f * t;
            }
            vfma(u6_6, a1.z, dm[2]);
            { const float t = vdot(sx6_6, dm[2]);
              dyl[2] = fmaf(0.632455528f, t, dyl[2]);
            }
            vfma(u6_6, a2.y, dm[3]);
            { const float t = vdot(sx6_6, dm[3]);
              dyl[3] = fmaf(-0.316227764f, t, dyl[3]);
            }
            vfma(u6_6, a0.w, dm[1]);
            { const float t = vdot(sx6_6, dm[1]);
              dyl[1] = fmaf(-0.316227764f, t, dyl[1]);
            }
            vfma(u6_7, a1.w, dm[2]);
            { const float t = vdot(sx6_7, dm[2]);
              dyl[3] = fmaf(0.547722578f, t, dyl[3]);
            }
            vfma(u6_7, a2.z, dm[3]);
            { const float t = vdot(sx6_7, dm[3]);
              dyl[2] = fmaf(0.547722578f, t, dyl[2]);
            }
            vfma(u6_8, a1.x, dm[1]);
            { const float t = vdot(sx6_8, dm[1]);
              dyl[1] = fmaf(-0.547722578f, t, dyl[1]);
            }
            vfma(u6_8, a2.w, dm[3]);
            { const float t = vdot(sx6_8, dm[3]);
              dyl[3] = fmaf(0.547722578f, t, dyl[3]);
            }
            BVec ds6 = vmul(x4, u6_4);
            vfma(ds6, x5, u6_5);
            vfma(ds6, x6, u6_6);
            vfma(ds6, x7, u6_7);
            vfma(ds6, x8, u6_8);
            if (gw) gw[6 * NQV] = ds6;
            dxp[4] = vmul(s6, u6_4);
            dxp[5] = vmul(s6, u6_5);
            dxp[6] = vmul(s6, u6_6);
            dxp[7] = vmul(s6, u6_7);
            dxp[8] = vmul(s6, u6_8);
            const BVec s8 = ss[8 * NQV];  // path 8: l1=1 l2=1 -> L=1
            const BVec sx8_1 = vmul(s8, x1);
            BVec u8_1; vzero(u8_1);
            const BVec sx8_2 = vmul(s8, x2);
            BVec u8_2; vzero(u8_2);
            const BVec sx8_3 = vmul(s8, x3);
            BVec u8_3; vzero(u8_3);
            const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
            vfma(u8_2, a3.x, dm[4]);
            { const float t = vdot(sx8_2, dm[4]);
              dyl[3] = fmaf(0.707106769f, t, dyl[3]);
            }
            vfma(u8_1, a3.z, dm[5]);
            { const float t = vdot(sx8_1, dm[5]);
              dyl[3] = fmaf(-0.707106769f, t, dyl[3]);
            }
            const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
            vfma(u8_1, a4.x, dm[6]);
            { const float t = vdot(sx8_1, dm[6]);
              dyl[2] = fmaf(0.707106769f, t, dyl[2]);
            }
            vfma(u8_3, a3.y, dm[4]);
            { const float t = vdot(sx8_3, dm[4]);
              dyl[2] = fmaf(-0.707106769f, t, dyl[2]);
            }
            vfma(u8_3, a3.w, dm[5]);
            { const float t = vdot(sx8_3, dm[5]);
              dyl[1] = fmaf(0.707106769f, t, dyl[1]);
            }
            vfma(u8_2, a4.y, dm[6]);
            { const float t = vdot(sx8_2, dm[6]);
              dyl[1] = fmaf(-0.707106769f, t, dyl[1]);
            }
            BVec ds8 = vmul(x1, u8_1);
            vfma(ds8, x2, u8_2);
            vfma(ds8, x3, u8_3);
            if (gw) gw[8 * NQV] = ds8;
            dxp[1] = vmul(s8, u8_1);
            dxp[2] = vmul(s8, u8_2);
            dxp[3] = vmul(s8, u8_3);
            const BVec s10 = ss[10 * NQV];  // path 10: l1=0 l2=2 -> L=2
            const BVec sx10_0 = vmul(s10, x0);
            BVec u10_0; vzero(u10_0);
            vfma(u10_0, a4.z, dm[7]);
            { const float t = vdot(sx10_0, dm[7]);
              dyl[4] = 1.0f * t;
            }
            vfma(u10_0, a4.w, dm[8]);
            { const float t = vdot(sx10_0, dm[8]);
              dyl[5] = 1.0f * t;
            }
            const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
            vfma(u10_0, a5.x, dm[9]);
            { const float t = vdot(sx10_0, dm[9]);
              dyl[6] = 1.0f * t;
            }
            vfma(u10_0, a5.y, dm[10]);
            { const float t = vdot(sx10_0, dm[10]);
              dyl[7] = 1.0f * t;
            }
            vfma(u10_0, a5.z, dm[11]);
            { const float t = vdot(sx10_0, dm[11]);
              dyl[8] = 1.0f * t;
            }
            BVec ds10 = vmul(x0, u10_0);
            if (gw) gw[10 * NQV] = ds10;
            vfma(dxp[0], s10, u10_0);
            const BVec s17 = ss[17 * NQV];  // path 17: l1=3 l2=2 -> L=2
            const BVec sx17_9 = vmul(s17, x9);
            BVec u17_9; vzero(u17_9);
            const BVec sx17_10 = vmul(s17, x10);
            BVec u17_10; vzero(u17_10);
            const BVec sx17_11 = vmul(s17, x11);
            BVec u17_11; vzero(u17_11);
            const BVec sx17_12 = vmul(s17, x12);
            BVec u17_12; vzero(u17_12);
            const BVec sx17_13 = vmul(s17, x13);
            BVec u17_13; vzero(u17_13);
            const BVec sx17_14 = vmul(s17, x14);
            BVec u17_14; vzero(u17_14);
            const BVec sx17_15 = vmul(s17, x15);
            BVec u17_15; vzero(u17_15);
            vfma(u17_9, a5.w, dm[12]);
            { const float t = vdot(sx17_9, dm[12]);
              dyl[5] = fmaf(0.422577113f, t, dyl[5]);
            }
            const float4 a7 = *reinterpret_cast<const float4*>(As + 28);
            vfma(u17_9, a7.y, dm[13]);
            { const float t = vdot(sx17_9, dm[13]);
              dyl[4] = fmaf(-0.422577113f, t, dyl[4]);
            }
            const float4 a8 = *reinterpret_cast<const float4*>(As + 32);
            vfma(u17_10, a8.z, dm[14]);
            { const float t = vdot(sx17_10, dm[14]);
              dyl[8] = fmaf(0.597614288f, t, dyl[8]);
            }
            const float4 a9 = *reinterpret_cast<const float4*>(As + 36);
            vfma(u17_9, a9.z, dm[15]);
            { const float t = vdot(sx17_9, dm[15]);
              dyl[8] = fmaf(0.422577113f, t, dyl[8]);
            }
            const float4 a10 = *reinterpret_cast<const float4*>(As + 40);
            vfma(u17_9, a10.w, dm[16]);
            { const float t = vdot(sx17_9, dm[16]);
              dyl[7] = fmaf(-0.422577113f, t, dyl[7]);
            }
            const float4 a6 = *reinterpret_cast<const float4*>(As + 24);
            vfma(u17_11, a6.x, dm[12]);
            { const float t = vdot(sx17_11, dm[12]);
              dyl[5] = fmaf(0.327326834f, t, dyl[5]);
            }
            vfma(u17_11, a7.z, dm[13]);
            { const float t = vdot(sx17_11, dm[13]);
              dyl[4] = fmaf(-0.327326834f, t, dyl[4]);
            }
            vfma(u17_11, a8.w, dm[14]);
            { const float t = vdot(sx17_11, dm[14]);
              dyl[7] = fmaf(0.377964467f, t, dyl[7]);
            }
            vfma(u17_11, a9.w, dm[15]);
            { const float t = vdot(sx17_11, dm[15]);
              dyl[6] = fmaf(-0.377964467f, t, dyl[6]);
              dyl[8] = fmaf(-0.327326834f, t, dyl[8]);
            }
            const float4 a11 = *reinterpret_cast<const float4*>(As + 44);
            vfma(u17_10, a11.x, dm[16]);
            { const float t = vdot(sx17_10, dm[16]);
              dyl[6] = fmaf(-0.597614288f, t, dyl[6]);
            }
            vfma(u17_12, a6.y, dm[12]);
            { const float t = vdot(sx17_12, dm[12]);
              dyl[8] = fmaf(0.267261237f, t, dyl[8]);
            }
            vfma(u17_12, a7.w, dm[13]);
            { const float t = vdot(sx17_12, dm[13]);
              dyl[7] = fmaf(-0.534522474f, t, dyl[7]);
            }
            vfma(u17_13, a9.x, dm[14]);
            { const float t = vdot(sx17_13, dm[14]);
              dyl[5] = fmaf(-0.377964467f, t, dyl[5]);
            }
            vfma(u17_12, a10.x, dm[15]);
            { const float t = vdot(sx17_12, dm[15]);
              dyl[5] = fmaf(0.534522474f, t, dyl[5]);
            }
            vfma(u17_11, a11.y, dm[16]);
            { const float t = vdot(sx17_11, dm[16]);
              dyl[7] = fmaf(0.327326834f, t, dyl[7]);
            }
            vfma(u17_13, a6.z, dm[12]);
            { const float t = vdot(sx17_13, dm[12]);
              dyl[7] = fmaf(-0.327326834f, t, dyl[7]);
            }
            vfma(u17_13, a8.x, dm[13]);
            { const float t = vdot(sx17_13, dm[13]);
              dyl[6] = fmaf(0.377964467f, t, dyl[6]);
              dyl[8] = fmaf(-0.327326834f, t, dyl[8]);
            }
            vfma(u17_14, a9.y, dm[14]);
            { const float t = vdot(sx17_14, dm[14]);
              dyl[4] = fmaf(-0.597614288f, t, dyl[4]);
            }
            vfma(u17_13, a10.y, dm[15]);
            { const float t = vdot(sx17_13, dm[15]);
              dyl[4] = fmaf(0.327326834f, t, dyl[4]);
            }
            vfma(u17_12, a11.z, dm[16]);
            { const float t = vdot(sx17_12, dm[16]);
              dyl[4] = fmaf(-0.267261237f, t, dyl[4]);
            }
            vfma(u17_14, a6.w, dm[12]);
            { const float t = vdot(sx17_14, dm[12]);
              dyl[6] = fmaf(0.597614288f, t, dyl[6]);
            }
            vfma(u17_15, a8.y, dm[13]);
            { const float t = vdot(sx17_15, dm[13]);
              dyl[8] = fmaf(-0.422577113f, t, dyl[8]);
            }
            vfma(u17_15, a10.z, dm[15]);
            { const float t = vdot(sx17_15, dm[15]);
              dyl[4] = fmaf(-0.422577113f, t, dyl[4]);
            }
            vfma(u17_13, a11.w, dm[16]);
            { const float t = vdot(sx17_13, dm[16]);
              dyl[5] = fmaf(0.327326834f, t, dyl[5]);
            }
            vfma(u17_15, a7.x, dm[12]);
            { const float t = vdot(sx17_15, dm[12]);
              dyl[7] = fmaf(0.422577113f, t, dyl[7]);
            }
            const float4 a12 = *reinterpret_cast<const float4*>(As + 48);
            vfma(u17_15, a12.x, dm[16]);
            { const float t = vdot(sx17_15, dm[16]);
              dyl[5] = fmaf(0.422577113f, t, dyl[5]);
            }
            BVec ds17 = vmul(x9, u17_9);
            vfma(ds17, x10, u17_10);
            vfma(ds17, x11, u17_11);
            vfma(ds17, x12, u17_12);
            vfma(ds17, x13, u17_13);
            vfma(ds17, x14, u17_14);
            vfma(ds17, x15, u17_15);
            if (gw) gw[17 * NQV] = ds17;
            dxp[9] = vmul(s17, u17_9);
            dxp[10] = vmul(s17, u17_10);
            dxp[11] = vmul(s17, u17_11);
            dxp[12] = vmul(s17, u17_12);
            dxp[13] = vmul(s17, u17_13);
            dxp[14] = vmul(s17, u17_14);
            dxp[15] = vmul(s17, u17_15);
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
            const BVec x9 = xs[9 * NQV];
            const BVec x10 = xs[10 * NQV];
            const BVec x11 = xs[11 * NQV];
            const BVec x12 = xs[12 * NQV];
            const BVec x13 = xs[13 * NQV];
            const BVec x14 = xs[14 * NQV];
            const BVec x15 = xs[15 * NQV];
            const BVec s1 = ss[1 * NQV];  // path 1: l1=1 l2=1 -> L=0
            const BVec sx1_1 = vmul(s1, x1);
            BVec u1_1; vzero(u1_1);
            const BVec sx1_2 = vmul(s1, x2);
            BVec u1_2; vzero(u1_2);
            const BVec sx1_3 = vmul(s1, x3);
            BVec u1_3; vzero(u1_3);
            const float4 a13 = *reinterpret_cast<const float4*>(As + 52);
            vfma(u1_1, a13.x, dm[0]);
            { const float t = vdot(sx1_1, dm[0]);
              dyl[1] = 0.577350259f * t;
            }
            vfma(u1_2, a13.y, dm[0]);
            { const float t = vdot(sx1_2, dm[0]);
              dyl[2] = 0.577350259f * t;
            }
            vfma(u1_3, a13.z, dm[0]);
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
            const BVec s3 = ss[3 * NQV];  // path 3: l1=0 l2=1 -> L=1
            const BVec sx3_0 = vmul(s3, x0);
            BVec u3_0; vzero(u3_0);
            vfma(u3_0, a13.w, dm[1]);
            { const float t = vdot(sx3_0, dm[1]);
              dyl[1] = fmaf(1.0f, t, dyl[1]);
            }
            const float4 a14 = *reinterpret_cast<const float4*>(As + 56);
            vfma(u3_0, a14.x, dm[2]);
            { const float t = vdot(sx3_0, dm[2]);
              dyl[2] = fmaf(1.0f, t, dyl[2]);
            }
            vfma(u3_0, a14.y, dm[3]);
            { const float t = vdot(sx3_0, dm[3]);
              dyl[3] = fmaf(1.0f, t, dyl[3]);
            }
            BVec ds3 = vmul(x0, u3_0);
            if (gw) gw[3 * NQV] = ds3;
            dxp[0] = vmul(s3, u3_0);
            const BVec s5 = ss[5 * NQV];  // path 5: l1=1 l2=2 -> L=1
            const BVec sx5_1 = vmul(s5, x1);
            BVec u5_1; vzero(u5_1);
            const BVec sx5_2 = vmul(s5, x2);
            BVec u5_2; vzero(u5_2);
            const BVec sx5_3 = vmul(s5, x3);
            BVec u5_3; vzero(u5_3);
            vfma(u5_1, a14.z, dm[4]);
            { const float t = vdot(sx5_1, dm[4]);
              dyl[6] = 0.316227764f * t;
              dyl[8] = 0.547722578f * t;
            }
            const float4 a15 = *reinterpret_cast<const float4*>(As + 60);
            vfma(u5_1, a15.y, dm[5]);
            { const float t = vdot(sx5_1, dm[5]);
              dyl[5] = -0.547722578f * t;
            }
            const float4 a16 = *reinterpret_cast<const float4*>(As + 64);
            vfma(u5_1, a16.x, dm[6]);
            { const float t = vdot(sx5_1, dm[6]);
              dyl[4] = -0.547722578f * t;
            }
            vfma(u5_2, a14.w, dm[4]);
            { const float t = vdot(sx5_2, dm[4]);
              dyl[5] = fmaf(-0.547722578f, t, dyl[5]);
            }
            vfma(u5_2, a15.z, dm[5]);
            { const float t = vdot(sx5_2, dm[5]);
              dyl[6] = fmaf(-0.632455528f, t, dyl[6]);
            }
            vfma(u5_2, a16.y, dm[6]);
            { const float t = vdot(sx5_2, dm[6]);
              dyl[7] = -0.547722578f * t;
            }
            vfma(u5_3, a15.x, dm[4]);
            { const float t = vdot(sx5_3, dm[4]);
              dyl[4] = fmaf(-0.547722578f, t, dyl[4]);
            }
            vfma(u5_3, a15.w, dm[5]);
            { const float t = vdot(sx5_3, dm[5]);
              dyl[7] = fmaf(-0.547722578f, t, dyl[7]);
            }
            vfma(u5_3, a16.z, dm[6]);
            { const float t = vdot(sx5_3, dm[6]);
              dyl[6] = fmaf(0.316227764f, t, dyl[6]);
              dyl[8] = fmaf(-0.547722578f, t, dyl[8]);
            }
            BVec ds5 = vmul(x1, u5_1);
            vfma(ds5, x2, u5_2);
            vfma(ds5, x3, u5_3);
            if (gw) gw[5 * NQV] = ds5;
            vfma(dxp[1], s5, u5_1);
            vfma(dxp[2], s5, u5_2);
            vfma(dxp[3], s5, u5_3);
            const BVec s14 = ss[14 * NQV];  // path 14: l1=3 l2=1 -> L=2
            const BVec sx14_9 = vmul(s14, x9);
            BVec u14_9; vzero(u14_9);
            const BVec sx14_10 = vmul(s14, x10);
            BVec u14_10; vzero(u14_10);
            const BVec sx14_11 = vmul(s14, x11);
            BVec u14_11; vzero(u14_11);
            const BVec sx14_12 = vmul(s14, x12);
            BVec u14_12; vzero(u14_12);
            const BVec sx14_13 = vmul(s14, x13);
            BVec u14_13; vzero(u14_13);
            const BVec sx14_14 = vmul(s14, x14);
            BVec u14_14; vzero(u14_14);
            const BVec sx14_15 = vmul(s14, x15);
            BVec u14_15; vzero(u14_15);
            vfma(u14_9, a16.w, dm[7]);
            { const float t = vdot(sx14_9, dm[7]);
              dyl[3] = fmaf(0.597614288f, t, dyl[3]);
            }
            const float4 a18 = *reinterpret_cast<const float4*>(As + 72);
            vfma(u14_10, a18.x, dm[8]);
            { const float t = vdot(sx14_10, dm[8]);
              dyl[3] = fmaf(0.487950027f, t, dyl[3]);
            }
            const float4 a19 = *reinterpret_cast<const float4*>(As + 76);
            vfma(u14_11, a19.x, dm[9]);
            { const float t = vdot(sx14_11, dm[9]);
              dyl[1] = fmaf(0.534522474f, t, dyl[1]);
            }
            vfma(u14_10, a19.w, dm[10]);
            { const float t = vdot(sx14_10, dm[10]);
              dyl[1] = fmaf(0.487950027f, t, dyl[1]);
            }
            const float4 a20 = *reinterpret_cast<const float4*>(As + 80);
            vfma(u14_9, a20.w, dm[11]);
            { const float t = vdot(sx14_9, dm[11]);
              dyl[1] = fmaf(0.597614288f, t, dyl[1]);
            }
            const float4 a17 = *reinterpret_cast<const float4*>(As + 68);
            vfma(u14_10, a17.x, dm[7]);
            { const float t = vdot(sx14_10, dm[7]);
              dyl[2] = fmaf(0.487950027f, t, dyl[2]);
            }
            vfma(u14_11, a18.y, dm[8]);
            { const float t = vdot(sx14_11, dm[8]);
              dyl[2] = fmaf(0.617213428f, t, dyl[2]);
            }
            vfma(u14_12, a19.y, dm[9]);
            { const float t = vdot(sx14_12, dm[9]);
              dyl[2] = fmaf(0.654653668f, t, dyl[2]);
            }
            vfma(u14_12, a20.x, dm[10]);
            { const float t = vdot(sx14_12, dm[10]);
              dyl[3] = fmaf(-0.377964467f, t, dyl[3]);
            }
            const float4 a21 = *reinterpret_cast<const float4*>(As + 84);
            vfma(u14_11, a21.x, dm[11]);
            { const float t = vdot(sx14_11, dm[11]);
              dyl[1] = fmaf(0.154303357f, t, dyl[1]);
            }
            vfma(u14_11, a17.y, dm[7]);
            { const float t = vdot(sx14_11, dm[7]);
              dyl[3] = fmaf(-0.154303357f, t, dyl[3]);
            }
            vfma(u14_12, a18.z, dm[8]);
            { const float t = vdot(sx14_12, dm[8]);
              dyl[1] = fmaf(-0.377964467f, t, dyl[1]);
            }
            vfma(u14_13, a19.z, dm[9]);
            { const float t = vdot(sx14_13, dm[9]);
              dyl[3] = fmaf(0.534522474f, t, dyl[3]);
            }
            vfma(u14_13, a20.y, dm[10]);
            { const float t = vdot(sx14_13, dm[10]);
              dyl[2] = fmaf(0.617213428f, t, dyl[2]);
            }
            vfma(u14_13, a21.y, dm[11]);
            { const float t = vdot(sx14_13, dm[11]);
              dyl[3] = fmaf(-0.154303357f, t, dyl[3]);
            }
            vfma(u14_13, a17.z, dm[7]);
            { const float t = vdot(sx14_13, dm[7]);
              dyl[1] = fmaf(-0.154303357f, t, dyl[1]);
            }
            vfma(u14_14, a18.w, dm[8]);
            { const float t = vdot(sx14_14, dm[8]);
              dyl[1] = fmaf(-0.487950027f, t, dyl[1]);
            }
            vfma(u14_14, a20.z, dm[10]);
            { const float t = vdot(sx14_14, dm[10]);
              dyl[3] = fmaf(0.487950027f, t, dyl[3]);
            }
            vfma(u14_14, a21.z, dm[11]);
            { const float t = vdot(sx14_14, dm[11]);
              dyl[2] = fmaf(0.487950027f, t, dyl[2]);
            }
            vfma(u14_15, a17.w, dm[7]);
            { const float t = vdot(sx14_15, dm[7]);
              dyl[1] = fmaf(-0.597614288f, t, dyl[1]);
            }
            vfma(u14_15, a21.w, dm[11]);
            { const float t = vdot(sx14_15, dm[11]);
              dyl[3] = fmaf(0.597614288f, t, dyl[3]);
            }
            BVec ds14 = vmul(x9, u14_9);
            vfma(ds14, x10, u14_10);
            vfma(ds14, x11, u14_11);
            vfma(ds14, x12, u14_12);
            vfma(ds14, x13, u14_13);
            vfma(ds14, x14, u14_14);
            vfma(ds14, x15, u14_15);
            if (gw) gw[14 * NQV] = ds14;
            dxp[9] = vmul(s14, u14_9);
            dxp[10] = vmul(s14, u14_10);
            dxp[11] = vmul(s14, u14_11);
            dxp[12] = vmul(s14, u14_12);
            dxp[13] = vmul(s14, u14_13);
            dxp[14] = vmul(s14, u14_14);
            dxp[15] = vmul(s14, u14_15);
            const BVec s15 = ss[15 * NQV];  // path 15: l1=1 l2=2 -> L=2
            const BVec sx15_1 = vmul(s15, x1);
            BVec u15_1; vzero(u15_1);
            const BVec sx15_2 = vmul(s15, x2);
            BVec u15_2; vzero(u15_2);
            const BVec sx15_3 = vmul(s15, x3);
            BVec u15_3; vzero(u15_3);
            const float4 a22 = *reinterpret_cast<const float4*>(As + 88);
            vfma(u15_1, a22.x, dm[12]);
            { const float t = vdot(sx15_1, dm[12]);
              dyl[5] = fmaf(0.408248305f, t, dyl[5]);
            }
            vfma(u15_1, a22.w, dm[13]);
            { const float t = vdot(sx15_1, dm[13]);
              dyl[4] = fmaf(-0.408248305f, t, dyl[4]);
            }
            const float4 a23 = *reinterpret_cast<const float4*>(As + 92);
            vfma(u15_1, a23.z, dm[14]);
            { const float t = vdot(sx15_1, dm[14]);
              dyl[7] = fmaf(-0.707106769f, t, dyl[7]);
            }
            const float4 a24 = *reinterpret_cast<const float4*>(As + 96);
            vfma(u15_1, a24.x, dm[15]);
            { const float t = vdot(sx15_1, dm[15]);
              dyl[6] = fmaf(0.707106769f, t, dyl[6]);
              dyl[8] = fmaf(-0.408248305f, t, dyl[8]);
            }
            vfma(u15_1, a24.w, dm[16]);
            { const float t = vdot(sx15_1, dm[16]);
              dyl[7] = fmaf(0.408248305f, t, dyl[7]);
            }
            vfma(u15_2, a22.y, dm[12]);
            { const float t = vdot(sx15_2, dm[12]);
              dyl[8] = fmaf(0.816496611f, t, dyl[8]);
            }
            vfma(u15_2, a23.x, dm[13]);
            { const float t = vdot(sx15_2, dm[13]);
              dyl[7] = fmaf(0.408248305f, t, dyl[7]);
            }
            vfma(u15_3, a23.w, dm[14]);
            { const float t = vdot(sx15_3, dm[14]);
              dyl[5] = fmaf(0.707106769f, t, dyl[5]);
            }
            vfma(u15_2, a24.y, dm[15]);
            { const float t = vdot(sx15_2, dm[15]);
              dyl[5] = fmaf(-0.408248305f, t, dyl[5]);
            }
            const float4 a25 = *reinterpret_cast<const float4*>(As + 100);
            vfma(u15_2, a25.x, dm[16]);
            { const float t = vdot(sx15_2, dm[16]);
              dyl[4] = fmaf(-0.816496611f, t, dyl[4]);
            }
            vfma(u15_3, a22.z, dm[12]);
            { const float t = vdot(sx15_3, dm[12]);
              dyl[7] = fmaf(-0.408248305f, t, dyl[7]);
            }
            vfma(u15_3, a23.y, dm[13]);
            { const float t = vdot(sx15_3, dm[13]);
              dyl[6] = fmaf(-0.707106769f, t, dyl[6]);
              dyl[8] = fmaf(-0.408248305f, t, dyl[8]);
            }
            vfma(u15_3, a24.z, dm[15]);
            { const float t = vdot(sx15_3, dm[15]);
              dyl[4] = fmaf(0.408248305f, t, dyl[4]);
            }
            vfma(u15_3, a25.y, dm[16]);
            { const float t = vdot(sx15_3, dm[16]);
              dyl[5] = fmaf(0.408248305f, t, dyl[5]);
            }
            BVec ds15 = vmul(x1, u15_1);
            vfma(ds15, x2, u15_2);
            vfma(ds15, x3, u15_3);
            if (gw) gw[15 * NQV] = ds15;
            vfma(dxp[1], s15, u15_1);
            vfma(dxp[2], s15, u15_2);
            vfma(dxp[3], s15, u15_3);
            vzero(dxp[4]);
            vzero(dxp[5]);
            vzero(dxp[6]);
            vzero(dxp[7]);
            vzero(dxp[8]);
            dyl[0] = 0.f;
            dyl[9] = 0.f;
            dyl[10] = 0.f;
            dyl[11] = 0.f;
            dyl[12] = 0.f;
            dyl[13] = 0.f;
            dyl[14] = 0.f;
            dyl[15] = 0.f;
        } break;
        case 2: {
            const BVec x4 = xs[4 * NQV];
            const BVec x5 = xs[5 * NQV];
            const BVec x6 = xs[6 * NQV];
            const BVec x7 = xs[7 * NQV];
            const BVec x8 = xs[8 * NQV];
            const BVec x9 = xs[9 * NQV];
            const BVec x10 = xs[10 * NQV];
            const BVec x11 = xs[11 * NQV];
            const BVec x12 = xs[12 * NQV];
            const BVec x13 = xs[13 * NQV];
            const BVec x14 = xs[14 * NQV];
            const BVec x15 = xs[15 * NQV];
            const BVec s2 = ss[2 * NQV];  // path 2: l1=2 l2=2 -> L=0
            const BVec sx2_4 = vmul(s2, x4);
            BVec u2_4; vzero(u2_4);
            const BVec sx2_5 = vmul(s2, x5);
            BVec u2_5; vzero(u2_5);
            const BVec sx2_6 = vmul(s2, x6);
            BVec u2_6; vzero(u2_6);
            const BVec sx2_7 = vmul(s2, x7);
            BVec u2_7; vzero(u2_7);
            const BVec sx2_8 = vmul(s2, x8);
            BVec u2_8; vzero(u2_8);
            const float4 a26 = *reinterpret_cast<const float4*>(As + 104);
            vfma(u2_4, a26.x, dm[0]);
            { const float t = vdot(sx2_4, dm[0]);
              dyl[4] = 0.44721359f * t;
            }
            vfma(u2_5, a26.y, dm[0]);
            { const float t = vdot(sx2_5, dm[0]);
              dyl[5] = 0.44721359f * t;
            }
            vfma(u2_6, a26.z, dm[0]);
            { const float t = vdot(sx2_6, dm[0]);
              dyl[6] = 0.44721359f * t;
            }
            vfma(u2_7, a26.w, dm[0]);
            { const float t = vdot(sx2_7, dm[0]);
              dyl[7] = 0.44721359f * t;
            }
            const float4 a27 = *reinterpret_cast<const float4*>(As + 108);
            vfma(u2_8, a27.x, dm[0]);
            { const float t = vdot(sx2_8, dm[0]);
              dyl[8] = 0.44721359f * t;
            }
            BVec ds2 = vmul(x4, u2_4);
            vfma(ds2, x5, u2_5);
            vfma(ds2, x6, u2_6);
            vfma(ds2, x7, u2_7);
            vfma(ds2, x8, u2_8);
            if (gw) gw[2 * NQV] = ds2;
            dxp[4] = vmul(s2, u2_4);
            dxp[5] = vmul(s2, u2_5);
            dxp[6] = vmul(s2, u2_6);
            dxp[7] = vmul(s2, u2_7);
            dxp[8] = vmul(s2, u2_8);
            const BVec s7 = ss[7 * NQV];  // path 7: l1=3 l2=2 -> L=1
            const BVec sx7_9 = vmul(s7, x9);
            BVec u7_9; vzero(u7_9);
            const BVec sx7_10 = vmul(s7, x10);
            BVec u7_10; vzero(u7_10);
            const BVec sx7_11 = vmul(s7, x11);
            BVec u7_11; vzero(u7_11);
            const BVec sx7_12 = vmul(s7, x12);
            BVec u7_12; vzero(u7_12);
            const BVec sx7_13 = vmul(s7, x13);
            BVec u7_13; vzero(u7_13);
            const BVec sx7_14 = vmul(s7, x14);
            BVec u7_14; vzero(u7_14);
            const BVec sx7_15 = vmul(s7, x15);
            BVec u7_15; vzero(u7_15);
            vfma(u7_9, a27.y, dm[1]);
            { const float t = vdot(sx7_9, dm[1]);
              dyl[8] = fmaf(0.462910056f, t, dyl[8]);
            }
            const float4 a29 = *reinterpret_cast<const float4*>(As + 116);
            vfma(u7_10, a29.x, dm[2]);
            { const float t = vdot(sx7_10, dm[2]);
              dyl[4] = fmaf(0.377964467f, t, dyl[4]);
            }
            const float4 a30 = *reinterpret_cast<const float4*>(As + 120);
            vfma(u7_9, a30.y, dm[3]);
            { const float t = vdot(sx7_9, dm[3]);
              dyl[4] = fmaf(0.462910056f, t, dyl[4]);
            }
            vfma(u7_10, a27.z, dm[1]);
            { const float t = vdot(sx7_10, dm[1]);
              dyl[7] = fmaf(0.377964467f, t, dyl[7]);
            }
            vfma(u7_11, a29.y, dm[2]);
            { const float t = vdot(sx7_11, dm[2]);
              dyl[5] = fmaf(0.478091449f, t, dyl[5]);
            }
            vfma(u7_10, a30.z, dm[3]);
            { const float t = vdot(sx7_10, dm[3]);
              dyl[5] = fmaf(0.377964467f, t, dyl[5]);
            }
            vfma(u7_11, a27.w, dm[1]);
            { const float t = vdot(sx7_11, dm[1]);
              dyl[6] = fmaf(0.414039344f, t, dyl[6]);
              dyl[8] = fmaf(0.119522862f, t, dyl[8]);
            }
            vfma(u7_12, a29.z, dm[2]);
            { const float t = vdot(sx7_12, dm[2]);
              dyl[6] = fmaf(0.507092535f, t, dyl[6]);
            }
            vfma(u7_11, a30.w, dm[3]);
            { const float t = vdot(sx7_11, dm[3]);
              dyl[4] = fmaf(-0.119522862f, t, dyl[4]);
            }
            const float4 a28 = *reinterpret_cast<const float4*>(As + 112);
            vfma(u7_12, a28.x, dm[1]);
            { const float t = vdot(sx7_12, dm[1]);
              dyl[5] = fmaf(-0.292770028f, t, dyl[5]);
            }
            vfma(u7_13, a29.w, dm[2]);
            { const float t = vdot(sx7_13, dm[2]);
              dyl[7] = fmaf(0.478091449f, t, dyl[7]);
            }
            const float4 a31 = *reinterpret_cast<const float4*>(As + 124);
            vfma(u7_12, a31.x, dm[3]);
            { const float t = vdot(sx7_12, dm[3]);
              dyl[7] = fmaf(-0.292770028f, t, dyl[7]);
            }
            vfma(u7_13, a28.y, dm[1]);
            { const float t = vdot(sx7_13, dm[1]);
              dyl[4] = fmaf(-0.119522862f, t, dyl[4]);
            }
            vfma(u7_14, a30.x, dm[2]);
            { const float t = vdot(sx7_14, dm[2]);
              dyl[8] = fmaf(0.377964467f, t, dyl[8]);
            }
            vfma(u7_13, a31.y, dm[3]);
            { const float t = vdot(sx7_13, dm[3]);
              dyl[6] = fmaf(0.414039344f, t, dyl[6]);
              dyl[8] = fmaf(-0.119522862f, t, dyl[8]);
            }
            vfma(u7_14, a28.z, dm[1]);
            { const float t = vdot(sx7_14, dm[1]);
              dyl[5] = fmaf(-0.377964467f, t, dyl[5]);
            }
            vfma(u7_14, a31.z, dm[3]);
            { const float t = vdot(sx7_14, dm[3]);
              dyl[7] = fmaf(0.377964467f, t, dyl[7]);
            }
            vfma(u7_15, a28.w, dm[1]);
            { const float t = vdot(sx7_15, dm[1]);
              dyl[4] = fmaf(-0.462910056f, t, dyl[4]);
            }
            vfma(u7_15, a31.w, dm[3]);
            { const float t = vdot(sx7_15, dm[3]);
              dyl[8] = fmaf(0.462910056f, t, dyl[8]);
            }
            BVec ds7 = vmul(x9, u7_9);
            vfma(ds7, x10, u7_10);
            vfma(ds7, x11, u7_11);
            vfma(ds7, x12, u7_12);
            vfma(ds7, x13, u7_13);
            vfma(ds7, x14, u7_14);
            vfma(ds7, x15, u7_15);
            if (gw) gw[7 * NQV] = ds7;
            dxp[9] = vmul(s7, u7_9);
            dxp[10] = vmul(s7, u7_10);
            dxp[11] = vmul(s7, u7_11);
            dxp[12] = vmul(s7, u7_12);
            dxp[13] = vmul(s7, u7_13);
            dxp[14] = vmul(s7, u7_14);
            dxp[15] = vmul(s7, u7_15);
            const BVec s12 = ss[12 * NQV];  // path 12: l1=2 l2=0 -> L=2
            const BVec sx12_4 = vmul(s12, x4);
            BVec u12_4; vzero(u12_4);
            const BVec sx12_5 = vmul(s12, x5);
            BVec u12_5; vzero(u12_5);
            const BVec sx12_6 = vmul(s12, x6);
            BVec u12_6; vzero(u12_6);
            const BVec sx12_7 = vmul(s12, x7);
            BVec u12_7; vzero(u12_7);
            const BVec sx12_8 = vmul(s12, x8);
            BVec u12_8; vzero(u12_8);
            const float4 a32 = *reinterpret_cast<const float4*>(As + 128);
            vfma(u12_4, a32.x, dm[4]);
            { const float t = vdot(sx12_4, dm[4]);
              dyl[0] = 1.0f * t;
            }
            vfma(u12_5, a32.y, dm[5]);
            { const float t = vdot(sx12_5, dm[5]);
              dyl[0] = fmaf(1.0f, t, dyl[0]);
            }
            vfma(u12_6, a32.z, dm[6]);
            { const float t = vdot(sx12_6, dm[6]);
              dyl[0] = fmaf(1.0f, t, dyl[0]);
            }
            vfma(u12_7, a32.w, dm[7]);
            { const float t = vdot(sx12_7, dm[7]);
              dyl[0] = fmaf(1.0f, t, dyl[0]);
            }
            const float4 a33 = *reinterpret_cast<const float4*>(As + 132);
            vfma(u12_8, a33.x, dm[8]);
            { const float t = vdot(sx12_8, dm[8]);
              dyl[0] = fmaf(1.0f, t, dyl[0]);
            }
            BVec ds12 = vmul(x4, u12_4);
            vfma(ds12, x5, u12_5);
            vfma(ds12, x6, u12_6);
            vfma(ds12, x7, u12_7);
            vfma(ds12, x8, u12_8);
            if (gw) gw[12 * NQV] = ds12;
            vfma(dxp[4], s12, u12_4);
            vfma(dxp[5], s12, u12_5);
            vfma(dxp[6], s12, u12_6);
            vfma(dxp[7], s12, u12_7);
            vfma(dxp[8], s12, u12_8);
            const BVec s16 = ss[16 * NQV];  // path 16: l1=2 l2=1 -> L=2
            const BVec sx16_4 = vmul(s16, x4);
            BVec u16_4; vzero(u16_4);
            const BVec sx16_5 = vmul(s16, x5);
            BVec u16_5; vzero(u16_5);
            const BVec sx16_6 = vmul(s16, x6);
            BVec u16_6; vzero(u16_6);
            const BVec sx16_7 = vmul(s16, x7);
            BVec u16_7; vzero(u16_7);
            const BVec sx16_8 = vmul(s16, x8);
            BVec u16_8; vzero(u16_8);
            vfma(u16_5, a33.y, dm[9]);
            { const float t = vdot(sx16_5, dm[9]);
              dyl[1] = 0.408248305f * t;
            }
            const float4 a34 = *reinterpret_cast<const float4*>(As + 136);
            vfma(u16_4, a34.x, dm[10]);
            { const float t = vdot(sx16_4, dm[10]);
              dyl[1] = fmaf(-0.408248305f, t, dyl[1]);
            }
            const float4 a35 = *reinterpret_cast<const float4*>(As + 140);
            vfma(u16_5, a35.x, dm[11]);
            { const float t = vdot(sx16_5, dm[11]);
              dyl[3] = 0.707106769f * t;
            }
            vfma(u16_4, a35.z, dm[12]);
            { const float t = vdot(sx16_4, dm[12]);
              dyl[3] = fmaf(0.408248305f, t, dyl[3]);
            }
            const float4 a36 = *reinterpret_cast<const float4*>(As + 144);
            vfma(u16_4, a36.z, dm[13]);
            { const float t = vdot(sx16_4, dm[13]);
              dyl[2] = -0.816496611f * t;
            }
            vfma(u16_7, a33.z, dm[9]);
            { const float t = vdot(sx16_7, dm[9]);
              dyl[3] = fmaf(-0.408248305f, t, dyl[3]);
            }
            vfma(u16_6, a34.y, dm[10]);
            { const float t = vdot(sx16_6, dm[10]);
              dyl[3] = fmaf(-0.707106769f, t, dyl[3]);
            }
            vfma(u16_7, a35.y, dm[11]);
            { const float t = vdot(sx16_7, dm[11]);
              dyl[1] = fmaf(-0.707106769f, t, dyl[1]);
            }
            vfma(u16_5, a35.w, dm[12]);
            { const float t = vdot(sx16_5, dm[12]);
              dyl[2] = fmaf(-0.408248305f, t, dyl[2]);
            }
            vfma(u16_5, a36.w, dm[13]);
            { const float t = vdot(sx16_5, dm[13]);
              dyl[3] = fmaf(0.408248305f, t, dyl[3]);
            }
            vfma(u16_8, a33.w, dm[9]);
            { const float t = vdot(sx16_8, dm[9]);
              dyl[2] = fmaf(0.816496611f, t, dyl[2]);
            }
            vfma(u16_7, a34.z, dm[10]);
            { const float t = vdot(sx16_7, dm[10]);
              dyl[2] = fmaf(0.408248305f, t, dyl[2]);
            }
            vfma(u16_6, a36.x, dm[12]);
            { const float t = vdot(sx16_6, dm[12]);
              dyl[1] = fmaf(0.707106769f, t, dyl[1]);
            }
            const float4 a37 = *reinterpret_cast<const float4*>(As + 148);
            vfma(u16_7, a37.x, dm[13]);
            { const float t = vdot(sx16_7, dm[13]);
              dyl[1] = fmaf(0.408248305f, t, dyl[1]);
            }
            vfma(u16_8, a34.w, dm[10]);
            { const float t = vdot(sx16_8, dm[10]);
              dyl[3] = fmaf(-0.408248305f, t, dyl[3]);
            }
            vfma(u16_8, a36.y, dm[12]);
            { const float t = vdot(sx16_8, dm[12]);
              dyl[1] = fmaf(-0.408248305f, t, dyl[1]);
            }
            BVec ds16 = vmul(x4, u16_4);
            vfma(ds16, x5, u16_5);
            vfma(ds16, x6, u16_6);
            vfma(ds16, x7, u16_7);
            vfma(ds16, x8, u16_8);
            if (gw) gw[16 * NQV] = ds16;
            vfma(dxp[4], s16, u16_4);
            vfma(dxp[5], s16, u16_5);
            vfma(dxp[6], s16, u16_6);
            vfma(dxp[7], s16, u16_7);
            vfma(dxp[8], s16, u16_8);
            vzero(dxp[0]);
            vzero(dxp[1]);
            vzero(dxp[2]);
            vzero(dxp[3]);
            dyl[9] = 0.f;
            dyl[10] = 0.f;
            dyl[11] = 0.f;
            dyl[12] = 0.f;
            dyl[13] = 0.f;
            dyl[14] = 0.f;
            dyl[15] = 0.f;
        } break;
        case 3: {
            const BVec x1 = xs[1 * NQV];
            const BVec x2 = xs[2 * NQV];
            const BVec x3 = xs[3 * NQV];
            const BVec x4 = xs[4 * NQV];
            const BVec x5 = xs[5 * NQV];
            const BVec x6 = xs[6 * NQV];
            const BVec x7 = xs[7 * NQV];
            const BVec x8 = xs[8 * NQV];
            const BVec s4 = ss[4 * NQV];  // path 4: l1=1 l2=0 -> L=1
            const BVec sx4_1 = vmul(s4, x1);
            BVec u4_1; vzero(u4_1);
            const BVec sx4_2 = vmul(s4, x2);
            BVec u4_2; vzero(u4_2);
            const BVec sx4_3 = vmul(s4, x3);
            BVec u4_3; vzero(u4_3);
            const float4 a38 = *reinterpret_cast<const float4*>(As + 152);
            vfma(u4_1, a38.x, dm[0]);
            { const float t = vdot(sx4_1, dm[0]);
              dyl[0] = 1.0f * t;
            }
            vfma(u4_2, a38.y, dm[1]);
            { const float t = vdot(sx4_2, dm[1]);
              dyl[0] = fmaf(1.0f, t, dyl[0]);
            }
            vfma(u4_3, a38.z, dm[2]);
            { const float t = vdot(sx4_3, dm[2]);
              dyl[0] = fmaf(1.0f, t, dyl[0]);
            }
            BVec ds4 = vmul(x1, u4_1);
            vfma(ds4, x2, u4_2);
            vfma(ds4, x3, u4_3);
            if (gw) gw[4 * NQV] = ds4;
            dxp[1] = vmul(s4, u4_1);
            dxp[2] = vmul(s4, u4_2);
            dxp[3] = vmul(s4, u4_3);
            const BVec s9 = ss[9 * NQV];  // path 9: l1=2 l2=2 -> L=1
            const BVec sx9_4 = vmul(s9, x4);
            BVec u9_4; vzero(u9_4);
            const BVec sx9_5 = vmul(s9, x5);
            BVec u9_5; vzero(u9_5);
            const BVec sx9_6 = vmul(s9, x6);
            BVec u9_6; vzero(u9_6);
            const BVec sx9_7 = vmul(s9, x7);
            BVec u9_7; vzero(u9_7);
            const BVec sx9_8 = vmul(s9, x8);
            BVec u9_8; vzero(u9_8);
            vfma(u9_4, a38.w, dm[3]);
            { const float t = vdot(sx9_4, dm[3]);
              dyl[5] = 0.316227764f * t;
            }
            const float4 a40 = *reinterpret_cast<const float4*>(As + 160);
            vfma(u9_4, a40.x, dm[4]);
            { const float t = vdot(sx9_4, dm[4]);
              dyl[8] = 0.632455528f * t;
            }
            const float4 a41 = *reinterpret_cast<const float4*>(As + 164);
            vfma(u9_4, a41.x, dm[5]);
            { const float t = vdot(sx9_4, dm[5]);
              dyl[7] = -0.316227764f * t;
            }
            const float4 a39 = *reinterpret_cast<const float4*>(As + 156);
            vfma(u9_5, a39.x, dm[3]);
            { const float t = vdot(sx9_5, dm[3]);
              dyl[4] = -0.316227764f * t;
            }
            vfma(u9_5, a40.y, dm[4]);
            { const float t = vdot(sx9_5, dm[4]);
              dyl[7] = fmaf(0.316227764f, t, dyl[7]);
            }
            vfma(u9_5, a41.y, dm[5]);
            { const float t = vdot(sx9_5, dm[5]);
              dyl[6] = -0.547722578f * t;
              dyl[8] = fmaf(-0.316227764f, t, dyl[8]);
            }
            vfma(u9_6, a39.y, dm[3]);
            { const float t = vdot(sx9_6, dm[3]);
              dyl[7] = fmaf(-0.547722578f, t, dyl[7]);
            }
            vfma(u9_7, a40.z, dm[4]);
            { const float t = vdot(sx9_7, dm[4]);
              dyl[5] = fmaf(-0.316227764f, t, dyl[5]);
            }
            vfma(u9_6, a41.z, dm[5]);
            { const float t = vdot(sx9_6, dm[5]);
              dyl[5] = fmaf(0.547722578f, t, dyl[5]);
            }
            vfma(u9_7, a39.z, dm[3]);
            { const float t = vdot(sx9_7, dm[3]);
              dyl[6] = fmaf(0.547722578f, t, dyl[6]);
              dyl[8] = fmaf(-0.316227764f, t, dyl[8]);
            }
            vfma(u9_8, a40.w, dm[4]);
            { const float t = vdot(sx9_8, dm[4]);
              dyl[4] = fmaf(-0.632455528f, t, dyl[4]);
            }
            vfma(u9_7, a41.w, dm[5]);
            { const float t = vdot(sx9_7, dm[5]);
              dyl[4] = fmaf(0.316227764f, t, dyl[4]);
            }
            vfma(u9_8, a39.w, dm[3]);
            { const float t = vdot(sx9_8, dm[3]);
              dyl[7] = fmaf(0.316227764f, t, dyl[7]);
            }
            const float4 a42 = *reinterpret_cast<const float4*>(As + 168);
            vfma(u9_8, a42.x, dm[5]);
            { const float t = vdot(sx9_8, dm[5]);
              dyl[5] = fmaf(0.316227764f, t, dyl[5]);
            }
            BVec ds9 = vmul(x4, u9_4);
            vfma(ds9, x5, u9_5);
            vfma(ds9, x6, u9_6);
            vfma(ds9, x7, u9_7);
            vfma(ds9, x8, u9_8);
            if (gw) gw[9 * NQV] = ds9;
            dxp[4] = vmul(s9, u9_4);
            dxp[5] = vmul(s9, u9_5);
            dxp[6] = vmul(s9, u9_6);
            dxp[7] = vmul(s9, u9_7);
            dxp[8] = vmul(s9, u9_8);
            const BVec s11 = ss[11 * NQV];  // path 11: l1=1 l2=1 -> L=2
            const BVec sx11_1 = vmul(s11, x1);
            BVec u11_1; vzero(u11_1);
            const BVec sx11_2 = vmul(s11, x2);
            BVec u11_2; vzero(u11_2);
            const BVec sx11_3 = vmul(s11, x3);
            BVec u11_3; vzero(u11_3);
            vfma(u11_1, a42.y, dm[6]);
            { const float t = vdot(sx11_1, dm[6]);
              dyl[3] = 0.707106769f * t;
            }
            vfma(u11_1, a42.w, dm[7]);
            { const float t = vdot(sx11_1, dm[7]);
              dyl[2] = 0.707106769f * t;
            }
            const float4 a43 = *reinterpret_cast<const float4*>(As + 172);
            vfma(u11_1, a43.y, dm[8]);
            { const float t = vdot(sx11_1, dm[8]);
              dyl[1] = -0.408248305f * t;
            }
            const float4 a44 = *reinterpret_cast<const float4*>(As + 176);
            vfma(u11_2, a44.x, dm[9]);
            { const float t = vdot(sx11_2, dm[9]);
              dyl[3] = fmaf(0.707106769f, t, dyl[3]);
            }
            vfma(u11_1, a44.z, dm[10]);
            { const float t = vdot(sx11_1, dm[10]);
              dyl[1] = fmaf(-0.707106769f, t, dyl[1]);
            }
            vfma(u11_3, a42.z, dm[6]);
            { const float t = vdot(sx11_3, dm[6]);
              dyl[1] = fmaf(0.707106769f, t, dyl[1]);
            }
            vfma(u11_2, a43.x, dm[7]);
            { const float t = vdot(sx11_2, dm[7]);
              dyl[1] = fmaf(0.707106769f, t, dyl[1]);
            }
            vfma(u11_2, a43.z, dm[8]);
            { const float t = vdot(sx11_2, dm[8]);
              dyl[2] = fmaf(0.816496611f, t, dyl[2]);
            }
            vfma(u11_3, a44.y, dm[9]);
            { const float t = vdot(sx11_3, dm[9]);
              dyl[2] = fmaf(0.707106769f, t, dyl[2]);
            }
            vfma(u11_3, a44.w, dm[10]);
            { const float t = vdot(sx11_3, dm[10]);
              dyl[3] = fmaf(0.707106769f, t, dyl[3]);
            }
            vfma(u11_3, a43.w, dm[8]);
            { const float t = vdot(sx11_3, dm[8]);
              dyl[3] = fmaf(-0.408248305f, t, dyl[3]);
            }
            BVec ds11 = vmul(x1, u11_1);
            vfma(ds11, x2, u11_2);
            vfma(ds11, x3, u11_3);
            if (gw) gw[11 * NQV] = ds11;
            vfma(dxp[1], s11, u11_1);
            vfma(dxp[2], s11, u11_2);
            vfma(dxp[3], s11, u11_3);
            const BVec s13 = ss[13 * NQV];  // path 13: l1=2 l2=2 -> L=2
            const BVec sx13_4 = vmul(s13, x4);
            BVec u13_4; vzero(u13_4);
            const BVec sx13_5 = vmul(s13, x5);
            BVec u13_5; vzero(u13_5);
            const BVec sx13_6 = vmul(s13, x6);
            BVec u13_6; vzero(u13_6);
            const BVec sx13_7 = vmul(s13, x7);
            BVec u13_7; vzero(u13_7);
            const BVec sx13_8 = vmul(s13, x8);
            BVec u13_8; vzero(u13_8);
            const float4 a45 = *reinterpret_cast<const float4*>(As + 180);
            vfma(u13_4, a45.x, dm[11]);
            { const float t = vdot(sx13_4, dm[11]);
              dyl[6] = fmaf(0.534522474f, t, dyl[6]);
            }
            const float4 a46 = *reinterpret_cast<const float4*>(As + 184);
            vfma(u13_4, a46.x, dm[12]);
            { const float t = vdot(sx13_4, dm[12]);
              dyl[7] = fmaf(-0.462910056f, t, dyl[7]);
            }
            const float4 a47 = *reinterpret_cast<const float4*>(As + 188);
            vfma(u13_4, a47.y, dm[13]);
            { const float t = vdot(sx13_4, dm[13]);
              dyl[4] = fmaf(0.534522474f, t, dyl[4]);
            }
            const float4 a48 = *reinterpret_cast<const float4*>(As + 192);
            vfma(u13_4, a48.z, dm[14]);
            { const float t = vdot(sx13_4, dm[14]);
              dyl[5] = fmaf(-0.462910056f, t, dyl[5]);
            }
            const float4 a49 = *reinterpret_cast<const float4*>(As + 196);
            vfma(u13_5, a49.w, dm[15]);
            { const float t = vdot(sx13_5, dm[15]);
              dyl[5] = fmaf(0.462910056f, t, dyl[5]);
            }
            vfma(u13_5, a45.y, dm[11]);
            { const float t = vdot(sx13_5, dm[11]);
              dyl[7] = fmaf(-0.462910056f, t, dyl[7]);
            }
            vfma(u13_5, a46.y, dm[12]);
            { const float t = vdot(sx13_5, dm[12]);
              dyl[6] = fmaf(-0.267261237f, t, dyl[6]);
              dyl[8] = fmaf(0.462910056f, t, dyl[8]);
            }
            vfma(u13_5, a47.z, dm[13]);
            { const float t = vdot(sx13_5, dm[13]);
              dyl[5] = fmaf(-0.267261237f, t, dyl[5]);
            }
            vfma(u13_5, a48.w, dm[14]);
            { const float t = vdot(sx13_5, dm[14]);
              dyl[4] = fmaf(-0.462910056f, t, dyl[4]);
            }
            const float4 a50 = *reinterpret_cast<const float4*>(As + 200);
            vfma(u13_6, a50.x, dm[15]);
            { const float t = vdot(sx13_6, dm[15]);
              dyl[8] = fmaf(0.534522474f, t, dyl[8]);
            }
            vfma(u13_6, a45.z, dm[11]);
            { const float t = vdot(sx13_6, dm[11]);
              dyl[4] = fmaf(0.534522474f, t, dyl[4]);
            }
            vfma(u13_6, a46.z, dm[12]);
            { const float t = vdot(sx13_6, dm[12]);
              dyl[5] = fmaf(-0.267261237f, t, dyl[5]);
            }
            vfma(u13_6, a47.w, dm[13]);
            { const float t = vdot(sx13_6, dm[13]);
              dyl[6] = fmaf(-0.534522474f, t, dyl[6]);
            }
            vfma(u13_6, a49.x, dm[14]);
            { const float t = vdot(sx13_6, dm[14]);
              dyl[7] = fmaf(-0.267261237f, t, dyl[7]);
            }
            vfma(u13_7, a50.y, dm[15]);
            { const float t = vdot(sx13_7, dm[15]);
              dyl[7] = fmaf(-0.462910056f, t, dyl[7]);
            }
            vfma(u13_7, a45.w, dm[11]);
            { const float t = vdot(sx13_7, dm[11]);
              dyl[5] = fmaf(-0.462910056f, t, dyl[5]);
            }
            vfma(u13_7, a46.w, dm[12]);
            { const float t = vdot(sx13_7, dm[12]);
              dyl[4] = fmaf(-0.462910056f, t, dyl[4]);
            }
            vfma(u13_7, a48.x, dm[13]);
            { const float t = vdot(sx13_7, dm[13]);
              dyl[7] = fmaf(-0.267261237f, t, dyl[7]);
            }
            vfma(u13_7, a49.y, dm[14]);
            { const float t = vdot(sx13_7, dm[14]);
              dyl[6] = fmaf(-0.267261237f, t, dyl[6]);
              dyl[8] = fmaf(-0.462910056f, t, dyl[8]);
            }
            vfma(u13_8, a50.z, dm[15]);
            { const float t = vdot(sx13_8, dm[15]);
              dyl[6] = fmaf(0.534522474f, t, dyl[6]);
            }
            vfma(u13_8, a47.x, dm[12]);
            { const float t = vdot(sx13_8, dm[12]);
              dyl[5] = fmaf(0.462910056f, t, dyl[5]);
            }
            vfma(u13_8, a48.y, dm[13]);
            { const float t = vdot(sx13_8, dm[13]);
              dyl[8] = fmaf(0.534522474f, t, dyl[8]);
            }
            vfma(u13_8, a49.z, dm[14]);
            { const float t = vdot(sx13_8, dm[14]);
              dyl[7] = fmaf(-0.462910056f, t, dyl[7]);
            }
            BVec ds13 = vmul(x4, u13_4);
            vfma(ds13, x5, u13_5);
            vfma(ds13, x6, u13_6);
            vfma(ds13, x7, u13_7);
            vfma(ds13, x8, u13_8);
            if (gw) gw[13 * NQV] = ds13;
            vfma(dxp[4], s13, u13_4);
            vfma(dxp[5], s13, u13_5);
            vfma(dxp[6], s13, u13_6);
            vfma(dxp[7], s13, u13_7);
            vfma(dxp[8], s13, u13_8);
            vzero(dxp[0]);
            vzero(dxp[9]);
            vzero(dxp[10]);
            vzero(dxp[11]);
            vzero(dxp[12]);
            vzero(dxp[13]);
            vzero(dxp[14]);
            vzero(dxp[15]);
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
        const EVec x4 = xs[4 * NQV];
        const EVec x5 = xs[5 * NQV];
        const EVec x6 = xs[6 * NQV];
        const EVec x7 = xs[7 * NQV];
        const EVec x8 = xs[8 * NQV];
        const EVec x9 = xs[9 * NQV];
        const EVec x10 = xs[10 * NQV];
        const EVec x11 = xs[11 * NQV];
        const EVec x12 = xs[12 * NQV];
        const EVec x13 = xs[13 * NQV];
        const EVec x14 = xs[14 * NQV];
        const EVec x15 = xs[15 * NQV];
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
        const float4 a13 = *reinterpret_cast<const float4*>(As + 52);
        vfma(u1_1, a13.x, d1_1);
        { const float t = vdot(sx1_1, d1_1);
          dyl[1] = 0.577350259f * t;
        }
        vfma(u1_2, a13.y, d1_1);
        { const float t = vdot(sx1_2, d1_1);
          dyl[2] = 0.577350259f * t;
        }
        vfma(u1_3, a13.z, d1_1);
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
        const EVec s2 = ss[2 * NQV];  // path 2: l1=2 l2=2 -> L=0
        const EVec sx2_4 = vmul(s2, x4);
        EVec u2_4; vzero(u2_4);
        const EVec sx2_5 = vmul(s2, x5);
        EVec u2_5; vzero(u2_5);
        const EVec sx2_6 = vmul(s2, x6);
        EVec u2_6; vzero(u2_6);
        const EVec sx2_7 = vmul(s2, x7);
        EVec u2_7; vzero(u2_7);
        const EVec sx2_8 = vmul(s2, x8);
        EVec u2_8; vzero(u2_8);
        const EVec d2_2 = dms[2 * NQV];
        const float4 a26 = *reinterpret_cast<const float4*>(As + 104);
        vfma(u2_4, a26.x, d2_2);
        { const float t = vdot(sx2_4, d2_2);
          dyl[4] = 0.44721359f * t;
        }
        vfma(u2_5, a26.y, d2_2);
        { const float t = vdot(sx2_5, d2_2);
          dyl[5] = 0.44721359f * t;
        }
        vfma(u2_6, a26.z, d2_2);
        { const float t = vdot(sx2_6, d2_2);
          dyl[6] = 0.44721359f * t;
        }
        vfma(u2_7, a26.w, d2_2);
        { const float t = vdot(sx2_7, d2_2);
          dyl[7] = 0.44721359f * t;
        }
        const float4 a27 = *reinterpret_cast<const float4*>(As + 108);
        vfma(u2_8, a27.x, d2_2);
        { const float t = vdot(sx2_8, d2_2);
          dyl[8] = 0.44721359f * t;
        }
        EVec ds2 = vmul(x4, u2_4);
        vfma(ds2, x5, u2_5);
        vfma(ds2, x6, u2_6);
        vfma(ds2, x7, u2_7);
        vfma(ds2, x8, u2_8);
        if (gw) gw[2 * NQV] = ds2;
        dxp[4] = vmul(s2, u2_4);
        dxp[5] = vmul(s2, u2_5);
        dxp[6] = vmul(s2, u2_6);
        dxp[7] = vmul(s2, u2_7);
        dxp[8] = vmul(s2, u2_8);
        const EVec s3 = ss[3 * NQV];  // path 3: l1=0 l2=1 -> L=1
        const EVec sx3_0 = vmul(s3, x0);
        EVec u3_0; vzero(u3_0);
        const EVec d3_3 = dms[3 * NQV];
        vfma(u3_0, a13.w, d3_3);
        { const float t = vdot(sx3_0, d3_3);
          dyl[1] = fmaf(1.0f, t, dyl[1]);
        }
        const EVec d3_4 = dms[4 * NQV];
        const float4 a14 = *reinterpret_cast<const float4*>(As + 56);
        vfma(u3_0, a14.x, d3_4);
        { const float t = vdot(sx3_0, d3_4);
          dyl[2] = fmaf(1.0f, t, dyl[2]);
        }
        const EVec d3_5 = dms[5 * NQV];
        vfma(u3_0, a14.y, d3_5);
        { const float t = vdot(sx3_0, d3_5);
          dyl[3] = fmaf(1.0f, t, dyl[3]);
        }
        EVec ds3 = vmul(x0, u3_0);
        if (gw) gw[3 * NQV] = ds3;
        vfma(dxp[0], s3, u3_0);
        const EVec s4 = ss[4 * NQV];  // path 4: l1=1 l2=0 -> L=1
        const EVec sx4_1 = vmul(s4, x1);
        EVec u4_1; vzero(u4_1);
        const EVec sx4_2 = vmul(s4, x2);
        EVec u4_2; vzero(u4_2);
        const EVec sx4_3 = vmul(s4, x3);
        EVec u4_3; vzero(u4_3);
        const EVec d4_6 = dms[6 * NQV];
        const float4 a38 = *reinterpret_cast<const float4*>(As + 152);
        vfma(u4_1, a38.x, d4_6);
        { const float t = vdot(sx4_1, d4_6);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        const EVec d4_7 = dms[7 * NQV];
        vfma(u4_2, a38.y, d4_7);
        { const float t = vdot(sx4_2, d4_7);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        const EVec d4_8 = dms[8 * NQV];
        vfma(u4_3, a38.z, d4_8);
        { const float t = vdot(sx4_3, d4_8);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        EVec ds4 = vmul(x1, u4_1);
        vfma(ds4, x2, u4_2);
        vfma(ds4, x3, u4_3);
        if (gw) gw[4 * NQV] = ds4;
        vfma(dxp[1], s4, u4_1);
        vfma(dxp[2], s4, u4_2);
        vfma(dxp[3], s4, u4_3);
        const EVec s5 = ss[5 * NQV];  // path 5: l1=1 l2=2 -> L=1
        const EVec sx5_1 = vmul(s5, x1);
        EVec u5_1; vzero(u5_1);
        const EVec sx5_2 = vmul(s5, x2);
        EVec u5_2; vzero(u5_2);
        const EVec sx5_3 = vmul(s5, x3);
        EVec u5_3; vzero(u5_3);
        const EVec d5_9 = dms[9 * NQV];
        vfma(u5_1, a14.z, d5_9);
        { const float t = vdot(sx5_1, d5_9);
          dyl[6] = fmaf(0.316227764f, t, dyl[6]);
          dyl[8] = fmaf(0.547722578f, t, dyl[8]);
        }
        const EVec d5_10 = dms[10 * NQV];
        const float4 a15 = *reinterpret_cast<const float4*>(As + 60);
        vfma(u5_1, a15.y, d5_10);
        { const float t = vdot(sx5_1, d5_10);
          dyl[5] = fmaf(-0.547722578f, t, dyl[5]);
        }
        const EVec d5_11 = dms[11 * NQV];
        const float4 a16 = *reinterpret_cast<const float4*>(As + 64);
        vfma(u5_1, a16.x, d5_11);
        { const float t = vdot(sx5_1, d5_11);
          dyl[4] = fmaf(-0.547722578f, t, dyl[4]);
        }
        vfma(u5_2, a14.w, d5_9);
        { const float t = vdot(sx5_2, d5_9);
          dyl[5] = fmaf(-0.547722578f, t, dyl[5]);
        }
        vfma(u5_2, a15.z, d5_10);
        { const float t = vdot(sx5_2, d5_10);
          dyl[6] = fmaf(-0.632455528f, t, dyl[6]);
        }
        vfma(u5_2, a16.y, d5_11);
        { const float t = vdot(sx5_2, d5_11);
          dyl[7] = fmaf(-0.547722578f, t, dyl[7]);
        }
        vfma(u5_3, a15.x, d5_9);
        { const float t = vdot(sx5_3, d5_9);
          dyl[4] = fmaf(-0.547722578f, t, dyl[4]);
        }
        vfma(u5_3, a15.w, d5_10);
        { const float t = vdot(sx5_3, d5_10);
          dyl[7] = fmaf(-0.547722578f, t, dyl[7]);
        }
        vfma(u5_3, a16.z, d5_11);
        { const float t = vdot(sx5_3, d5_11);
          dyl[6] = fmaf(0.316227764f, t, dyl[6]);
          dyl[8] = fmaf(-0.547722578f, t, dyl[8]);
        }
        EVec ds5 = vmul(x1, u5_1);
        vfma(ds5, x2, u5_2);
        vfma(ds5, x3, u5_3);
        if (gw) gw[5 * NQV] = ds5;
        vfma(dxp[1], s5, u5_1);
        vfma(dxp[2], s5, u5_2);
        vfma(dxp[3], s5, u5_3);
        const EVec s6 = ss[6 * NQV];  // path 6: l1=2 l2=1 -> L=1
        const EVec sx6_4 = vmul(s6, x4);
        EVec u6_4; vzero(u6_4);
        const EVec sx6_5 = vmul(s6, x5);
        EVec u6_5; vzero(u6_5);
        const EVec sx6_6 = vmul(s6, x6);
        EVec u6_6; vzero(u6_6);
        const EVec sx6_7 = vmul(s6, x7);
        EVec u6_7; vzero(u6_7);
        const EVec sx6_8 = vmul(s6, x8);
        EVec u6_8; vzero(u6_8);
        const EVec d6_12 = dms[12 * NQV];
        vfma(u6_4, a0.y, d6_12);
        { const float t = vdot(sx6_4, d6_12);
          dyl[3] = fmaf(0.547722578f, t, dyl[3]);
        }
        const EVec d6_13 = dms[13 * NQV];
        const float4 a1 = *reinterpret_cast<const float4*>(As + 4);
        vfma(u6_5, a1.y, d6_13);
        { const float t = vdot(sx6_5, d6_13);
          dyl[1] = fmaf(0.547722578f, t, dyl[1]);
        }
        const EVec d6_14 = dms[14 * NQV];
        const float4 a2 = *reinterpret_cast<const float4*>(As + 8);
        vfma(u6_4, a2.x, d6_14);
        { const float t = vdot(sx6_4, d6_14);
          dyl[1] = fmaf(0.547722578f, t, dyl[1]);
        }
        vfma(u6_5, a0.z, d6_12);
        { const float t = vdot(sx6_5, d6_12);
          dyl[2] = fmaf(0.547722578f, t, dyl[2]);
        }
        vfma(u6_6, a1.z, d6_13);
        { const float t = vdot(sx6_6, d6_13);
          dyl[2] = fmaf(0.632455528f, t, dyl[2]);
        }
        vfma(u6_6, a2.y, d6_14);
        { const float t = vdot(sx6_6, d6_14);
          dyl[3] = fmaf(-0.316227764f, t, dyl[3]);
        }
        vfma(u6_6, a0.w, d6_12);
        { const float t = vdot(sx6_6, d6_12);
          dyl[1] = fmaf(-0.316227764f, t, dyl[1]);
        }
        vfma(u6_7, a1.w, d6_13);
        { const float t = vdot(sx6_7, d6_13);
          dyl[3] = fmaf(0.547722578f, t, dyl[3]);
        }
        vfma(u6_7, a2.z, d6_14);
        { const float t = vdot(sx6_7, d6_14);
          dyl[2] = fmaf(0.547722578f, t, dyl[2]);
        }
        vfma(u6_8, a1.x, d6_12);
        { const float t = vdot(sx6_8, d6_12);
          dyl[1] = fmaf(-0.547722578f, t, dyl[1]);
        }
        vfma(u6_8, a2.w, d6_14);
        { const float t = vdot(sx6_8, d6_14);
          dyl[3] = fmaf(0.547722578f, t, dyl[3]);
        }
        EVec ds6 = vmul(x4, u6_4);
        vfma(ds6, x5, u6_5);
        vfma(ds6, x6, u6_6);
        vfma(ds6, x7, u6_7);
        vfma(ds6, x8, u6_8);
        if (gw) gw[6 * NQV] = ds6;
        vfma(dxp[4], s6, u6_4);
        vfma(dxp[5], s6, u6_5);
        vfma(dxp[6], s6, u6_6);
        vfma(dxp[7], s6, u6_7);
        vfma(dxp[8], s6, u6_8);
        const EVec s7 = ss[7 * NQV];  // path 7: l1=3 l2=2 -> L=1
        const EVec sx7_9 = vmul(s7, x9);
        EVec u7_9; vzero(u7_9);
        const EVec sx7_10 = vmul(s7, x10);
        EVec u7_10; vzero(u7_10);
        const EVec sx7_11 = vmul(s7, x11);
        EVec u7_11; vzero(u7_11);
        const EVec sx7_12 = vmul(s7, x12);
        EVec u7_12; vzero(u7_12);
        const EVec sx7_13 = vmul(s7, x13);
        EVec u7_13; vzero(u7_13);
        const EVec sx7_14 = vmul(s7, x14);
        EVec u7_14; vzero(u7_14);
        const EVec sx7_15 = vmul(s7, x15);
        EVec u7_15; vzero(u7_15);
        const EVec d7_15 = dms[15 * NQV];
        vfma(u7_9, a27.y, d7_15);
        { const float t = vdot(sx7_9, d7_15);
          dyl[8] = fmaf(0.462910056f, t, dyl[8]);
        }
        const EVec d7_16 = dms[16 * NQV];
        const float4 a29 = *reinterpret_cast<const float4*>(As + 116);
        vfma(u7_10, a29.x, d7_16);
        { const float t = vdot(sx7_10, d7_16);
          dyl[4] = fmaf(0.377964467f, t, dyl[4]);
        }
        const EVec d7_17 = dms[17 * NQV];
        const float4 a30 = *reinterpret_cast<const float4*>(As + 120);
        vfma(u7_9, a30.y, d7_17);
        { const float t = vdot(sx7_9, d7_17);
          dyl[4] = fmaf(0.462910056f, t, dyl[4]);
        }
        vfma(u7_10, a27.z, d7_15);
        { const float t = vdot(sx7_10, d7_15);
          dyl[7] = fmaf(0.377964467f, t, dyl[7]);
        }
        vfma(u7_11, a29.y, d7_16);
        { const float t = vdot(sx7_11, d7_16);
          dyl[5] = fmaf(0.478091449f, t, dyl[5]);
        }
        vfma(u7_10, a30.z, d7_17);
        { const float t = vdot(sx7_10, d7_17);
          dyl[5] = fmaf(0.377964467f, t, dyl[5]);
        }
        vfma(u7_11, a27.w, d7_15);
        { const float t = vdot(sx7_11, d7_15);
          dyl[6] = fmaf(0.414039344f, t, dyl[6]);
          dyl[8] = fmaf(0.119522862f, t, dyl[8]);
        }
        vfma(u7_12, a29.z, d7_16);
        { const float t = vdot(sx7_12, d7_16);
          dyl[6] = fmaf(0.507092535f, t, dyl[6]);
        }
        vfma(u7_11, a30.w, d7_17);
        { const float t = vdot(sx7_11, d7_17);
          dyl[4] = fmaf(-0.119522862f, t, dyl[4]);
        }
        const float4 a28 = *reinterpret_cast<const float4*>(As + 112);
        vfma(u7_12, a28.x, d7_15);
        { const float t = vdot(sx7_12, d7_15);
          dyl[5] = fmaf(-0.292770028f, t, dyl[5]);
        }
        vfma(u7_13, a29.w, d7_16);
        { const float t = vdot(sx7_13, d7_16);
          dyl[7] = fmaf(0.478091449f, t, dyl[7]);
        }
        const float4 a31 = *reinterpret_cast<const float4*>(As + 124);
        vfma(u7_12, a31.x, d7_17);
        { const float t = vdot(sx7_12, d7_17);
          dyl[7] = fmaf(-0.292770028f, t, dyl[7]);
        }
        vfma(u7_13, a28.y, d7_15);
        { const float t = vdot(sx7_13, d7_15);
          dyl[4] = fmaf(-0.119522862f, t, dyl[4]);
        }
        vfma(u7_14, a30.x, d7_16);
        { const float t = vdot(sx7_14, d7_16);
          dyl[8] = fmaf(0.377964467f, t, dyl[8]);
        }
        vfma(u7_13, a31.y, d7_17);
        { const float t = vdot(sx7_13, d7_17);
          dyl[6] = fmaf(0.414039344f, t, dyl[6]);
          dyl[8] = fmaf(-0.119522862f, t, dyl[8]);
        }
        vfma(u7_14, a28.z, d7_15);
        { const float t = vdot(sx7_14, d7_15);
          dyl[5] = fmaf(-0.377964467f, t, dyl[5]);
        }
        vfma(u7_14, a31.z, d7_17);
        { const float t = vdot(sx7_14, d7_17);
          dyl[7] = fmaf(0.377964467f, t, dyl[7]);
        }
        vfma(u7_15, a28.w, d7_15);
        { const float t = vdot(sx7_15, d7_15);
          dyl[4] = fmaf(-0.462910056f, t, dyl[4]);
        }
        vfma(u7_15, a31.w, d7_17);
        { const float t = vdot(sx7_15, d7_17);
          dyl[8] = fmaf(0.462910056f, t, dyl[8]);
        }
        EVec ds7 = vmul(x9, u7_9);
        vfma(ds7, x10, u7_10);
        vfma(ds7, x11, u7_11);
        vfma(ds7, x12, u7_12);
        vfma(ds7, x13, u7_13);
        vfma(ds7, x14, u7_14);
        vfma(ds7, x15, u7_15);
        if (gw) gw[7 * NQV] = ds7;
        dxp[9] = vmul(s7, u7_9);
        dxp[10] = vmul(s7, u7_10);
        dxp[11] = vmul(s7, u7_11);
        dxp[12] = vmul(s7, u7_12);
        dxp[13] = vmul(s7, u7_13);
        dxp[14] = vmul(s7, u7_14);
        dxp[15] = vmul(s7, u7_15);
        const EVec s8 = ss[8 * NQV];  // path 8: l1=1 l2=1 -> L=1
        const EVec sx8_1 = vmul(s8, x1);
        EVec u8_1; vzero(u8_1);
        const EVec sx8_2 = vmul(s8, x2);
        EVec u8_2; vzero(u8_2);
        const EVec sx8_3 = vmul(s8, x3);
        EVec u8_3; vzero(u8_3);
        const EVec d8_18 = dms[18 * NQV];
        const float4 a3 = *reinterpret_cast<const float4*>(As + 12);
        vfma(u8_2, a3.x, d8_18);
        { const float t = vdot(sx8_2, d8_18);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        const EVec d8_19 = dms[19 * NQV];
        vfma(u8_1, a3.z, d8_19);
        { const float t = vdot(sx8_1, d8_19);
          dyl[3] = fmaf(-0.707106769f, t, dyl[3]);
        }
        const EVec d8_20 = dms[20 * NQV];
        const float4 a4 = *reinterpret_cast<const float4*>(As + 16);
        vfma(u8_1, a4.x, d8_20);
        { const float t = vdot(sx8_1, d8_20);
          dyl[2] = fmaf(0.707106769f, t, dyl[2]);
        }
        vfma(u8_3, a3.y, d8_18);
        { const float t = vdot(sx8_3, d8_18);
          dyl[2] = fmaf(-0.707106769f, t, dyl[2]);
        }
        vfma(u8_3, a3.w, d8_19);
        { const float t = vdot(sx8_3, d8_19);
          dyl[1] = fmaf(0.707106769f, t, dyl[1]);
        }
        vfma(u8_2, a4.y, d8_20);
        { const float t = vdot(sx8_2, d8_20);
          dyl[1] = fmaf(-0.707106769f, t, dyl[1]);
        }
        EVec ds8 = vmul(x1, u8_1);
        vfma(ds8, x2, u8_2);
        vfma(ds8, x3, u8_3);
        if (gw) gw[8 * NQV] = ds8;
        vfma(dxp[1], s8, u8_1);
        vfma(dxp[2], s8, u8_2);
        vfma(dxp[3], s8, u8_3);
        const EVec s9 = ss[9 * NQV];  // path 9: l1=2 l2=2 -> L=1
        const EVec sx9_4 = vmul(s9, x4);
        EVec u9_4; vzero(u9_4);
        const EVec sx9_5 = vmul(s9, x5);
        EVec u9_5; vzero(u9_5);
        const EVec sx9_6 = vmul(s9, x6);
        EVec u9_6; vzero(u9_6);
        const EVec sx9_7 = vmul(s9, x7);
        EVec u9_7; vzero(u9_7);
        const EVec sx9_8 = vmul(s9, x8);
        EVec u9_8; vzero(u9_8);
        const EVec d9_21 = dms[21 * NQV];
        vfma(u9_4, a38.w, d9_21);
        { const float t = vdot(sx9_4, d9_21);
          dyl[5] = fmaf(0.316227764f, t, dyl[5]);
        }
        const EVec d9_22 = dms[22 * NQV];
        const float4 a40 = *reinterpret_cast<const float4*>(As + 160);
        vfma(u9_4, a40.x, d9_22);
        { const float t = vdot(sx9_4, d9_22);
          dyl[8] = fmaf(0.632455528f, t, dyl[8]);
        }
        const EVec d9_23 = dms[23 * NQV];
        const float4 a41 = *reinterpret_cast<const float4*>(As + 164);
        vfma(u9_4, a41.x, d9_23);
        { const float t = vdot(sx9_4, d9_23);
          dyl[7] = fmaf(-0.316227764f, t, dyl[7]);
        }
        const float4 a39 = *reinterpret_cast<const float4*>(As + 156);
        vfma(u9_5, a39.x, d9_21);
        { const float t = vdot(sx9_5, d9_21);
          dyl[4] = fmaf(-0.316227764f, t, dyl[4]);
        }
        vfma(u9_5, a40.y, d9_22);
        { const float t = vdot(sx9_5, d9_22);
          dyl[7] = fmaf(0.316227764f, t, dyl[7]);
        }
        vfma(u9_5, a41.y, d9_23);
        { const float t = vdot(sx9_5, d9_23);
          dyl[6] = fmaf(-0.547722578f, t, dyl[6]);
          dyl[8] = fmaf(-0.316227764f, t, dyl[8]);
        }
        vfma(u9_6, a39.y, d9_21);
        { const float t = vdot(sx9_6, d9_21);
          dyl[7] = fmaf(-0.547722578f, t, dyl[7]);
        }
        vfma(u9_7, a40.z, d9_22);
        { const float t = vdot(sx9_7, d9_22);
          dyl[5] = fmaf(-0.316227764f, t, dyl[5]);
        }
        vfma(u9_6, a41.z, d9_23);
        { const float t = vdot(sx9_6, d9_23);
          dyl[5] = fmaf(0.547722578f, t, dyl[5]);
        }
        vfma(u9_7, a39.z, d9_21);
        { const float t = vdot(sx9_7, d9_21);
          dyl[6] = fmaf(0.547722578f, t, dyl[6]);
          dyl[8] = fmaf(-0.316227764f, t, dyl[8]);
        }
        vfma(u9_8, a40.w, d9_22);
        { const float t = vdot(sx9_8, d9_22);
          dyl[4] = fmaf(-0.632455528f, t, dyl[4]);
        }
        vfma(u9_7, a41.w, d9_23);
        { const float t = vdot(sx9_7, d9_23);
          dyl[4] = fmaf(0.316227764f, t, dyl[4]);
        }
        vfma(u9_8, a39.w, d9_21);
        { const float t = vdot(sx9_8, d9_21);
          dyl[7] = fmaf(0.316227764f, t, dyl[7]);
        }
        const float4 a42 = *reinterpret_cast<const float4*>(As + 168);
        vfma(u9_8, a42.x, d9_23);
        { const float t = vdot(sx9_8, d9_23);
          dyl[5] = fmaf(0.316227764f, t, dyl[5]);
        }
        EVec ds9 = vmul(x4, u9_4);
        vfma(ds9, x5, u9_5);
        vfma(ds9, x6, u9_6);
        vfma(ds9, x7, u9_7);
        vfma(ds9, x8, u9_8);
        if (gw) gw[9 * NQV] = ds9;
        vfma(dxp[4], s9, u9_4);
        vfma(dxp[5], s9, u9_5);
        vfma(dxp[6], s9, u9_6);
        vfma(dxp[7], s9, u9_7);
        vfma(dxp[8], s9, u9_8);
        const EVec s10 = ss[10 * NQV];  // path 10: l1=0 l2=2 -> L=2
        const EVec sx10_0 = vmul(s10, x0);
        EVec u10_0; vzero(u10_0);
        const EVec d10_24 = dms[24 * NQV];
        vfma(u10_0, a4.z, d10_24);
        { const float t = vdot(sx10_0, d10_24);
          dyl[4] = fmaf(1.0f, t, dyl[4]);
        }
        const EVec d10_25 = dms[25 * NQV];
        vfma(u10_0, a4.w, d10_25);
        { const float t = vdot(sx10_0, d10_25);
          dyl[5] = fmaf(1.0f, t, dyl[5]);
        }
        const EVec d10_26 = dms[26 * NQV];
        const float4 a5 = *reinterpret_cast<const float4*>(As + 20);
        vfma(u10_0, a5.x, d10_26);
        { const float t = vdot(sx10_0, d10_26);
          dyl[6] = fmaf(1.0f, t, dyl[6]);
        }
        const EVec d10_27 = dms[27 * NQV];
        vfma(u10_0, a5.y, d10_27);
        { const float t = vdot(sx10_0, d10_27);
          dyl[7] = fmaf(1.0f, t, dyl[7]);
        }
        const EVec d10_28 = dms[28 * NQV];
        vfma(u10_0, a5.z, d10_28);
        { const float t = vdot(sx10_0, d10_28);
          dyl[8] = fmaf(1.0f, t, dyl[8]);
        }
        EVec ds10 = vmul(x0, u10_0);
        if (gw) gw[10 * NQV] = ds10;
        vfma(dxp[0], s10, u10_0);
        const EVec s11 = ss[11 * NQV];  // path 11: l1=1 l2=1 -> L=2
        const EVec sx11_1 = vmul(s11, x1);
        EVec u11_1; vzero(u11_1);
        const EVec sx11_2 = vmul(s11, x2);
        EVec u11_2; vzero(u11_2);
        const EVec sx11_3 = vmul(s11, x3);
        EVec u11_3; vzero(u11_3);
        const EVec d11_29 = dms[29 * NQV];
        vfma(u11_1, a42.y, d11_29);
        { const float t = vdot(sx11_1, d11_29);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        const EVec d11_30 = dms[30 * NQV];
        vfma(u11_1, a42.w, d11_30);
        { const float t = vdot(sx11_1, d11_30);
          dyl[2] = fmaf(0.707106769f, t, dyl[2]);
        }
        const EVec d11_31 = dms[31 * NQV];
        const float4 a43 = *reinterpret_cast<const float4*>(As + 172);
        vfma(u11_1, a43.y, d11_31);
        { const float t = vdot(sx11_1, d11_31);
          dyl[1] = fmaf(-0.408248305f, t, dyl[1]);
        }
        const EVec d11_32 = dms[32 * NQV];
        const float4 a44 = *reinterpret_cast<const float4*>(As + 176);
        vfma(u11_2, a44.x, d11_32);
        { const float t = vdot(sx11_2, d11_32);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        const EVec d11_33 = dms[33 * NQV];
        vfma(u11_1, a44.z, d11_33);
        { const float t = vdot(sx11_1, d11_33);
          dyl[1] = fmaf(-0.707106769f, t, dyl[1]);
        }
        vfma(u11_3, a42.z, d11_29);
        { const float t = vdot(sx11_3, d11_29);
          dyl[1] = fmaf(0.707106769f, t, dyl[1]);
        }
        vfma(u11_2, a43.x, d11_30);
        { const float t = vdot(sx11_2, d11_30);
          dyl[1] = fmaf(0.707106769f, t, dyl[1]);
        }
        vfma(u11_2, a43.z, d11_31);
        { const float t = vdot(sx11_2, d11_31);
          dyl[2] = fmaf(0.816496611f, t, dyl[2]);
        }
        vfma(u11_3, a44.y, d11_32);
        { const float t = vdot(sx11_3, d11_32);
          dyl[2] = fmaf(0.707106769f, t, dyl[2]);
        }
        vfma(u11_3, a44.w, d11_33);
        { const float t = vdot(sx11_3, d11_33);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        vfma(u11_3, a43.w, d11_31);
        { const float t = vdot(sx11_3, d11_31);
          dyl[3] = fmaf(-0.408248305f, t, dyl[3]);
        }
        EVec ds11 = vmul(x1, u11_1);
        vfma(ds11, x2, u11_2);
        vfma(ds11, x3, u11_3);
        if (gw) gw[11 * NQV] = ds11;
        vfma(dxp[1], s11, u11_1);
        vfma(dxp[2], s11, u11_2);
        vfma(dxp[3], s11, u11_3);
        const EVec s12 = ss[12 * NQV];  // path 12: l1=2 l2=0 -> L=2
        const EVec sx12_4 = vmul(s12, x4);
        EVec u12_4; vzero(u12_4);
        const EVec sx12_5 = vmul(s12, x5);
        EVec u12_5; vzero(u12_5);
        const EVec sx12_6 = vmul(s12, x6);
        EVec u12_6; vzero(u12_6);
        const EVec sx12_7 = vmul(s12, x7);
        EVec u12_7; vzero(u12_7);
        const EVec sx12_8 = vmul(s12, x8);
        EVec u12_8; vzero(u12_8);
        const EVec d12_34 = dms[34 * NQV];
        const float4 a32 = *reinterpret_cast<const float4*>(As + 128);
        vfma(u12_4, a32.x, d12_34);
        { const float t = vdot(sx12_4, d12_34);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        const EVec d12_35 = dms[35 * NQV];
        vfma(u12_5, a32.y, d12_35);
        { const float t = vdot(sx12_5, d12_35);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        const EVec d12_36 = dms[36 * NQV];
        vfma(u12_6, a32.z, d12_36);
        { const float t = vdot(sx12_6, d12_36);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        const EVec d12_37 = dms[37 * NQV];
        vfma(u12_7, a32.w, d12_37);
        { const float t = vdot(sx12_7, d12_37);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        const EVec d12_38 = dms[38 * NQV];
        const float4 a33 = *reinterpret_cast<const float4*>(As + 132);
        vfma(u12_8, a33.x, d12_38);
        { const float t = vdot(sx12_8, d12_38);
          dyl[0] = fmaf(1.0f, t, dyl[0]);
        }
        EVec ds12 = vmul(x4, u12_4);
        vfma(ds12, x5, u12_5);
        vfma(ds12, x6, u12_6);
        vfma(ds12, x7, u12_7);
        vfma(ds12, x8, u12_8);
        if (gw) gw[12 * NQV] = ds12;
        vfma(dxp[4], s12, u12_4);
        vfma(dxp[5], s12, u12_5);
        vfma(dxp[6], s12, u12_6);
        vfma(dxp[7], s12, u12_7);
        vfma(dxp[8], s12, u12_8);
        const EVec s13 = ss[13 * NQV];  // path 13: l1=2 l2=2 -> L=2
        const EVec sx13_4 = vmul(s13, x4);
        EVec u13_4; vzero(u13_4);
        const EVec sx13_5 = vmul(s13, x5);
        EVec u13_5; vzero(u13_5);
        const EVec sx13_6 = vmul(s13, x6);
        EVec u13_6; vzero(u13_6);
        const EVec sx13_7 = vmul(s13, x7);
        EVec u13_7; vzero(u13_7);
        const EVec sx13_8 = vmul(s13, x8);
        EVec u13_8; vzero(u13_8);
        const EVec d13_39 = dms[39 * NQV];
        const float4 a45 = *reinterpret_cast<const float4*>(As + 180);
        vfma(u13_4, a45.x, d13_39);
        { const float t = vdot(sx13_4, d13_39);
          dyl[6] = fmaf(0.534522474f, t, dyl[6]);
        }
        const EVec d13_40 = dms[40 * NQV];
        const float4 a46 = *reinterpret_cast<const float4*>(As + 184);
        vfma(u13_4, a46.x, d13_40);
        { const float t = vdot(sx13_4, d13_40);
          dyl[7] = fmaf(-0.462910056f, t, dyl[7]);
        }
        const EVec d13_41 = dms[41 * NQV];
        const float4 a47 = *reinterpret_cast<const float4*>(As + 188);
        vfma(u13_4, a47.y, d13_41);
        { const float t = vdot(sx13_4, d13_41);
          dyl[4] = fmaf(0.534522474f, t, dyl[4]);
        }
        const EVec d13_42 = dms[42 * NQV];
        const float4 a48 = *reinterpret_cast<const float4*>(As + 192);
        vfma(u13_4, a48.z, d13_42);
        { const float t = vdot(sx13_4, d13_42);
          dyl[5] = fmaf(-0.462910056f, t, dyl[5]);
        }
        const EVec d13_43 = dms[43 * NQV];
        const float4 a49 = *reinterpret_cast<const float4*>(As + 196);
        vfma(u13_5, a49.w, d13_43);
        { const float t = vdot(sx13_5, d13_43);
          dyl[5] = fmaf(0.462910056f, t, dyl[5]);
        }
        vfma(u13_5, a45.y, d13_39);
        { const float t = vdot(sx13_5, d13_39);
          dyl[7] = fmaf(-0.462910056f, t, dyl[7]);
        }
        vfma(u13_5, a46.y, d13_40);
        { const float t = vdot(sx13_5, d13_40);
          dyl[6] = fmaf(-0.267261237f, t, dyl[6]);
          dyl[8] = fmaf(0.462910056f, t, dyl[8]);
        }
        vfma(u13_5, a47.z, d13_41);
        { const float t = vdot(sx13_5, d13_41);
          dyl[5] = fmaf(-0.267261237f, t, dyl[5]);
        }
        vfma(u13_5, a48.w, d13_42);
        { const float t = vdot(sx13_5, d13_42);
          dyl[4] = fmaf(-0.462910056f, t, dyl[4]);
        }
        const float4 a50 = *reinterpret_cast<const float4*>(As + 200);
        vfma(u13_6, a50.x, d13_43);
        { const float t = vdot(sx13_6, d13_43);
          dyl[8] = fmaf(0.534522474f, t, dyl[8]);
        }
        vfma(u13_6, a45.z, d13_39);
        { const float t = vdot(sx13_6, d13_39);
          dyl[4] = fmaf(0.534522474f, t, dyl[4]);
        }
        vfma(u13_6, a46.z, d13_40);
        { const float t = vdot(sx13_6, d13_40);
          dyl[5] = fmaf(-0.267261237f, t, dyl[5]);
        }
        vfma(u13_6, a47.w, d13_41);
        { const float t = vdot(sx13_6, d13_41);
          dyl[6] = fmaf(-0.534522474f, t, dyl[6]);
        }
        vfma(u13_6, a49.x, d13_42);
        { const float t = vdot(sx13_6, d13_42);
          dyl[7] = fmaf(-0.267261237f, t, dyl[7]);
        }
        vfma(u13_7, a50.y, d13_43);
        { const float t = vdot(sx13_7, d13_43);
          dyl[7] = fmaf(-0.462910056f, t, dyl[7]);
        }
        vfma(u13_7, a45.w, d13_39);
        { const float t = vdot(sx13_7, d13_39);
          dyl[5] = fmaf(-0.462910056f, t, dyl[5]);
        }
        vfma(u13_7, a46.w, d13_40);
        { const float t = vdot(sx13_7, d13_40);
          dyl[4] = fmaf(-0.462910056f, t, dyl[4]);
        }
        vfma(u13_7, a48.x, d13_41);
        { const float t = vdot(sx13_7, d13_41);
          dyl[7] = fmaf(-0.267261237f, t, dyl[7]);
        }
        vfma(u13_7, a49.y, d13_42);
        { const float t = vdot(sx13_7, d13_42);
          dyl[6] = fmaf(-0.267261237f, t, dyl[6]);
          dyl[8] = fmaf(-0.462910056f, t, dyl[8]);
        }
        vfma(u13_8, a50.z, d13_43);
        { const float t = vdot(sx13_8, d13_43);
          dyl[6] = fmaf(0.534522474f, t, dyl[6]);
        }
        vfma(u13_8, a47.x, d13_40);
        { const float t = vdot(sx13_8, d13_40);
          dyl[5] = fmaf(0.462910056f, t, dyl[5]);
        }
        vfma(u13_8, a48.y, d13_41);
        { const float t = vdot(sx13_8, d13_41);
          dyl[8] = fmaf(0.534522474f, t, dyl[8]);
        }
        vfma(u13_8, a49.z, d13_42);
        { const float t = vdot(sx13_8, d13_42);
          dyl[7] = fmaf(-0.462910056f, t, dyl[7]);
        }
        EVec ds13 = vmul(x4, u13_4);
        vfma(ds13, x5, u13_5);
        vfma(ds13, x6, u13_6);
        vfma(ds13, x7, u13_7);
        vfma(ds13, x8, u13_8);
        if (gw) gw[13 * NQV] = ds13;
        vfma(dxp[4], s13, u13_4);
        vfma(dxp[5], s13, u13_5);
        vfma(dxp[6], s13, u13_6);
        vfma(dxp[7], s13, u13_7);
        vfma(dxp[8], s13, u13_8);
        const EVec s14 = ss[14 * NQV];  // path 14: l1=3 l2=1 -> L=2
        const EVec sx14_9 = vmul(s14, x9);
        EVec u14_9; vzero(u14_9);
        const EVec sx14_10 = vmul(s14, x10);
        EVec u14_10; vzero(u14_10);
        const EVec sx14_11 = vmul(s14, x11);
        EVec u14_11; vzero(u14_11);
        const EVec sx14_12 = vmul(s14, x12);
        EVec u14_12; vzero(u14_12);
        const EVec sx14_13 = vmul(s14, x13);
        EVec u14_13; vzero(u14_13);
        const EVec sx14_14 = vmul(s14, x14);
        EVec u14_14; vzero(u14_14);
        const EVec sx14_15 = vmul(s14, x15);
        EVec u14_15; vzero(u14_15);
        const EVec d14_44 = dms[44 * NQV];
        vfma(u14_9, a16.w, d14_44);
        { const float t = vdot(sx14_9, d14_44);
          dyl[3] = fmaf(0.597614288f, t, dyl[3]);
        }
        const EVec d14_45 = dms[45 * NQV];
        const float4 a18 = *reinterpret_cast<const float4*>(As + 72);
        vfma(u14_10, a18.x, d14_45);
        { const float t = vdot(sx14_10, d14_45);
          dyl[3] = fmaf(0.487950027f, t, dyl[3]);
        }
        const EVec d14_46 = dms[46 * NQV];
        const float4 a19 = *reinterpret_cast<const float4*>(As + 76);
        vfma(u14_11, a19.x, d14_46);
        { const float t = vdot(sx14_11, d14_46);
          dyl[1] = fmaf(0.534522474f, t, dyl[1]);
        }
        const EVec d14_47 = dms[47 * NQV];
        vfma(u14_10, a19.w, d14_47);
        { const float t = vdot(sx14_10, d14_47);
          dyl[1] = fmaf(0.487950027f, t, dyl[1]);
        }
        const EVec d14_48 = dms[48 * NQV];
        const float4 a20 = *reinterpret_cast<const float4*>(As + 80);
        vfma(u14_9, a20.w, d14_48);
        { const float t = vdot(sx14_9, d14_48);
          dyl[1] = fmaf(0.597614288f, t, dyl[1]);
        }
        const float4 a17 = *reinterpret_cast<const float4*>(As + 68);
        vfma(u14_10, a17.x, d14_44);
        { const float t = vdot(sx14_10, d14_44);
          dyl[2] = fmaf(0.487950027f, t, dyl[2]);
        }
        vfma(u14_11, a18.y, d14_45);
        { const float t = vdot(sx14_11, d14_45);
          dyl[2] = fmaf(0.617213428f, t, dyl[2]);
        }
        vfma(u14_12, a19.y, d14_46);
        { const float t = vdot(sx14_12, d14_46);
          dyl[2] = fmaf(0.654653668f, t, dyl[2]);
        }
        vfma(u14_12, a20.x, d14_47);
        { const float t = vdot(sx14_12, d14_47);
          dyl[3] = fmaf(-0.377964467f, t, dyl[3]);
        }
        const float4 a21 = *reinterpret_cast<const float4*>(As + 84);
        vfma(u14_11, a21.x, d14_48);
        { const float t = vdot(sx14_11, d14_48);
          dyl[1] = fmaf(0.154303357f, t, dyl[1]);
        }
        vfma(u14_11, a17.y, d14_44);
        { const float t = vdot(sx14_11, d14_44);
          dyl[3] = fmaf(-0.154303357f, t, dyl[3]);
        }
        vfma(u14_12, a18.z, d14_45);
        { const float t = vdot(sx14_12, d14_45);
          dyl[1] = fmaf(-0.377964467f, t, dyl[1]);
        }
        vfma(u14_13, a19.z, d14_46);
        { const float t = vdot(sx14_13, d14_46);
          dyl[3] = fmaf(0.534522474f, t, dyl[3]);
        }
        vfma(u14_13, a20.y, d14_47);
        { const float t = vdot(sx14_13, d14_47);
          dyl[2] = fmaf(0.617213428f, t, dyl[2]);
        }
        vfma(u14_13, a21.y, d14_48);
        { const float t = vdot(sx14_13, d14_48);
          dyl[3] = fmaf(-0.154303357f, t, dyl[3]);
        }
        vfma(u14_13, a17.z, d14_44);
        { const float t = vdot(sx14_13, d14_44);
          dyl[1] = fmaf(-0.154303357f, t, dyl[1]);
        }
        vfma(u14_14, a18.w, d14_45);
        { const float t = vdot(sx14_14, d14_45);
          dyl[1] = fmaf(-0.487950027f, t, dyl[1]);
        }
        vfma(u14_14, a20.z, d14_47);
        { const float t = vdot(sx14_14, d14_47);
          dyl[3] = fmaf(0.487950027f, t, dyl[3]);
        }
        vfma(u14_14, a21.z, d14_48);
        { const float t = vdot(sx14_14, d14_48);
          dyl[2] = fmaf(0.487950027f, t, dyl[2]);
        }
        vfma(u14_15, a17.w, d14_44);
        { const float t = vdot(sx14_15, d14_44);
          dyl[1] = fmaf(-0.597614288f, t, dyl[1]);
        }
        vfma(u14_15, a21.w, d14_48);
        { const float t = vdot(sx14_15, d14_48);
          dyl[3] = fmaf(0.597614288f, t, dyl[3]);
        }
        EVec ds14 = vmul(x9, u14_9);
        vfma(ds14, x10, u14_10);
        vfma(ds14, x11, u14_11);
        vfma(ds14, x12, u14_12);
        vfma(ds14, x13, u14_13);
        vfma(ds14, x14, u14_14);
        vfma(ds14, x15, u14_15);
        if (gw) gw[14 * NQV] = ds14;
        vfma(dxp[9], s14, u14_9);
        vfma(dxp[10], s14, u14_10);
        vfma(dxp[11], s14, u14_11);
        vfma(dxp[12], s14, u14_12);
        vfma(dxp[13], s14, u14_13);
        vfma(dxp[14], s14, u14_14);
        vfma(dxp[15], s14, u14_15);
        const EVec s15 = ss[15 * NQV];  // path 15: l1=1 l2=2 -> L=2
        const EVec sx15_1 = vmul(s15, x1);
        EVec u15_1; vzero(u15_1);
        const EVec sx15_2 = vmul(s15, x2);
        EVec u15_2; vzero(u15_2);
        const EVec sx15_3 = vmul(s15, x3);
        EVec u15_3; vzero(u15_3);
        const EVec d15_49 = dms[49 * NQV];
        const float4 a22 = *reinterpret_cast<const float4*>(As + 88);
        vfma(u15_1, a22.x, d15_49);
        { const float t = vdot(sx15_1, d15_49);
          dyl[5] = fmaf(0.408248305f, t, dyl[5]);
        }
        const EVec d15_50 = dms[50 * NQV];
        vfma(u15_1, a22.w, d15_50);
        { const float t = vdot(sx15_1, d15_50);
          dyl[4] = fmaf(-0.408248305f, t, dyl[4]);
        }
        const EVec d15_51 = dms[51 * NQV];
        const float4 a23 = *reinterpret_cast<const float4*>(As + 92);
        vfma(u15_1, a23.z, d15_51);
        { const float t = vdot(sx15_1, d15_51);
          dyl[7] = fmaf(-0.707106769f, t, dyl[7]);
        }
        const EVec d15_52 = dms[52 * NQV];
        const float4 a24 = *reinterpret_cast<const float4*>(As + 96);
        vfma(u15_1, a24.x, d15_52);
        { const float t = vdot(sx15_1, d15_52);
          dyl[6] = fmaf(0.707106769f, t, dyl[6]);
          dyl[8] = fmaf(-0.408248305f, t, dyl[8]);
        }
        const EVec d15_53 = dms[53 * NQV];
        vfma(u15_1, a24.w, d15_53);
        { const float t = vdot(sx15_1, d15_53);
          dyl[7] = fmaf(0.408248305f, t, dyl[7]);
        }
        vfma(u15_2, a22.y, d15_49);
        { const float t = vdot(sx15_2, d15_49);
          dyl[8] = fmaf(0.816496611f, t, dyl[8]);
        }
        vfma(u15_2, a23.x, d15_50);
        { const float t = vdot(sx15_2, d15_50);
          dyl[7] = fmaf(0.408248305f, t, dyl[7]);
        }
        vfma(u15_3, a23.w, d15_51);
        { const float t = vdot(sx15_3, d15_51);
          dyl[5] = fmaf(0.707106769f, t, dyl[5]);
        }
        vfma(u15_2, a24.y, d15_52);
        { const float t = vdot(sx15_2, d15_52);
          dyl[5] = fmaf(-0.408248305f, t, dyl[5]);
        }
        const float4 a25 = *reinterpret_cast<const float4*>(As + 100);
        vfma(u15_2, a25.x, d15_53);
        { const float t = vdot(sx15_2, d15_53);
          dyl[4] = fmaf(-0.816496611f, t, dyl[4]);
        }
        vfma(u15_3, a22.z, d15_49);
        { const float t = vdot(sx15_3, d15_49);
          dyl[7] = fmaf(-0.408248305f, t, dyl[7]);
        }
        vfma(u15_3, a23.y, d15_50);
        { const float t = vdot(sx15_3, d15_50);
          dyl[6] = fmaf(-0.707106769f, t, dyl[6]);
          dyl[8] = fmaf(-0.408248305f, t, dyl[8]);
        }
        vfma(u15_3, a24.z, d15_52);
        { const float t = vdot(sx15_3, d15_52);
          dyl[4] = fmaf(0.408248305f, t, dyl[4]);
        }
        vfma(u15_3, a25.y, d15_53);
        { const float t = vdot(sx15_3, d15_53);
          dyl[5] = fmaf(0.408248305f, t, dyl[5]);
        }
        EVec ds15 = vmul(x1, u15_1);
        vfma(ds15, x2, u15_2);
        vfma(ds15, x3, u15_3);
        if (gw) gw[15 * NQV] = ds15;
        vfma(dxp[1], s15, u15_1);
        vfma(dxp[2], s15, u15_2);
        vfma(dxp[3], s15, u15_3);
        const EVec s16 = ss[16 * NQV];  // path 16: l1=2 l2=1 -> L=2
        const EVec sx16_4 = vmul(s16, x4);
        EVec u16_4; vzero(u16_4);
        const EVec sx16_5 = vmul(s16, x5);
        EVec u16_5; vzero(u16_5);
        const EVec sx16_6 = vmul(s16, x6);
        EVec u16_6; vzero(u16_6);
        const EVec sx16_7 = vmul(s16, x7);
        EVec u16_7; vzero(u16_7);
        const EVec sx16_8 = vmul(s16, x8);
        EVec u16_8; vzero(u16_8);
        const EVec d16_54 = dms[54 * NQV];
        vfma(u16_5, a33.y, d16_54);
        { const float t = vdot(sx16_5, d16_54);
          dyl[1] = fmaf(0.408248305f, t, dyl[1]);
        }
        const EVec d16_55 = dms[55 * NQV];
        const float4 a34 = *reinterpret_cast<const float4*>(As + 136);
        vfma(u16_4, a34.x, d16_55);
        { const float t = vdot(sx16_4, d16_55);
          dyl[1] = fmaf(-0.408248305f, t, dyl[1]);
        }
        const EVec d16_56 = dms[56 * NQV];
        const float4 a35 = *reinterpret_cast<const float4*>(As + 140);
        vfma(u16_5, a35.x, d16_56);
        { const float t = vdot(sx16_5, d16_56);
          dyl[3] = fmaf(0.707106769f, t, dyl[3]);
        }
        const EVec d16_57 = dms[57 * NQV];
        vfma(u16_4, a35.z, d16_57);
        { const float t = vdot(sx16_4, d16_57);
          dyl[3] = fmaf(0.408248305f, t, dyl[3]);
        }
        const EVec d16_58 = dms[58 * NQV];
        const float4 a36 = *reinterpret_cast<const float4*>(As + 144);
        vfma(u16_4, a36.z, d16_58);
        { const float t = vdot(sx16_4, d16_58);
          dyl[2] = fmaf(-0.816496611f, t, dyl[2]);
        }
        vfma(u16_7, a33.z, d16_54);
        { const float t = vdot(sx16_7, d16_54);
          dyl[3] = fmaf(-0.408248305f, t, dyl[3]);
        }
        vfma(u16_6, a34.y, d16_55);
        { const float t = vdot(sx16_6, d16_55);
          dyl[3] = fmaf(-0.707106769f, t, dyl[3]);
        }
        vfma(u16_7, a35.y, d16_56);
        { const float t = vdot(sx16_7, d16_56);
          dyl[1] = fmaf(-0.707106769f, t, dyl[1]);
        }
        vfma(u16_5, a35.w, d16_57);
        { const float t = vdot(sx16_5, d16_57);
          dyl[2] = fmaf(-0.408248305f, t, dyl[2]);
        }
        vfma(u16_5, a36.w, d16_58);
        { const float t = vdot(sx16_5, d16_58);
          dyl[3] = fmaf(0.408248305f, t, dyl[3]);
        }
        vfma(u16_8, a33.w, d16_54);
        { const float t = vdot(sx16_8, d16_54);
          dyl[2] = fmaf(0.816496611f, t, dyl[2]);
        }
        vfma(u16_7, a34.z, d16_55);
        { const float t = vdot(sx16_7, d16_55);
          dyl[2] = fmaf(0.408248305f, t, dyl[2]);
        }
        vfma(u16_6, a36.x, d16_57);
        { const float t = vdot(sx16_6, d16_57);
          dyl[1] = fmaf(0.707106769f, t, dyl[1]);
        }
        const float4 a37 = *reinterpret_cast<const float4*>(As + 148);
        vfma(u16_7, a37.x, d16_58);
        { const float t = vdot(sx16_7, d16_58);
          dyl[1] = fmaf(0.408248305f, t, dyl[1]);
        }
        vfma(u16_8, a34.w, d16_55);
        { const float t = vdot(sx16_8, d16_55);
          dyl[3] = fmaf(-0.408248305f, t, dyl[3]);
        }
        vfma(u16_8, a36.y, d16_57);
        { const float t = vdot(sx16_8, d16_57);
          dyl[1] = fmaf(-0.408248305f, t, dyl[1]);
        }
        EVec ds16 = vmul(x4, u16_4);
        vfma(ds16, x5, u16_5);
        vfma(ds16, x6, u16_6);
        vfma(ds16, x7, u16_7);
        vfma(ds16, x8, u16_8);
        if (gw) gw[16 * NQV] = ds16;
        vfma(dxp[4], s16, u16_4);
        vfma(dxp[5], s16, u16_5);
        vfma(dxp[6], s16, u16_6);
        vfma(dxp[7], s16, u16_7);
        vfma(dxp[8], s16, u16_8);
        const EVec s17 = ss[17 * NQV];  // path 17: l1=3 l2=2 -> L=2
        const EVec sx17_9 = vmul(s17, x9);
        EVec u17_9; vzero(u17_9);
        const EVec sx17_10 = vmul(s17, x10);
        EVec u17_10; vzero(u17_10);
        const EVec sx17_11 = vmul(s17, x11);
        EVec u17_11; vzero(u17_11);
        const EVec sx17_12 = vmul(s17, x12);
        EVec u17_12; vzero(u17_12);
        const EVec sx17_13 = vmul(s17, x13);
        EVec u17_13; vzero(u17_13);
        const EVec sx17_14 = vmul(s17, x14);
        EVec u17_14; vzero(u17_14);
        const EVec sx17_15 = vmul(s17, x15);
        EVec u17_15; vzero(u17_15);
        const EVec d17_59 = dms[59 * NQV];
        vfma(u17_9, a5.w, d17_59);
        { const float t = vdot(sx17_9, d17_59);
          dyl[5] = fmaf(0.422577113f, t, dyl[5]);
        }
        const EVec d17_60 = dms[60 * NQV];
        const float4 a7 = *reinterpret_cast<const float4*>(As + 28);
        vfma(u17_9, a7.y, d17_60);
        { const float t = vdot(sx17_9, d17_60);
          dyl[4] = fmaf(-0.422577113f, t, dyl[4]);
        }
        const EVec d17_61 = dms[61 * NQV];
        const float4 a8 = *reinterpret_cast<const float4*>(As + 32);
        vfma(u17_10, a8.z, d17_61);
        { const float t = vdot(sx17_10, d17_61);
          dyl[8] = fmaf(0.597614288f, t, dyl[8]);
        }
        const EVec d17_62 = dms[62 * NQV];
        const float4 a9 = *reinterpret_cast<const float4*>(As + 36);
        vfma(u17_9, a9.z, d17_62);
        { const float t = vdot(sx17_9, d17_62);
          dyl[8] = fmaf(0.422577113f, t, dyl[8]);
        }
        const EVec d17_63 = dms[63 * NQV];
        const float4 a10 = *reinterpret_cast<const float4*>(As + 40);
        vfma(u17_9, a10.w, d17_63);
        { const float t = vdot(sx17_9, d17_63);
          dyl[7] = fmaf(-0.422577113f, t, dyl[7]);
        }
        const float4 a6 = *reinterpret_cast<const float4*>(As + 24);
        vfma(u17_11, a6.x, d17_59);
        { const float t = vdot(sx17_11, d17_59);
          dyl[5] = fmaf(0.327326834f, t, dyl[5]);
        }
        vfma(u17_11, a7.z, d17_60);
        { const float t = vdot(sx17_11, d17_60);
          dyl[4] = fmaf(-0.327326834f, t, dyl[4]);
        }
        vfma(u17_11, a8.w, d17_61);
        { const float t = vdot(sx17_11, d17_61);
          dyl[7] = fmaf(0.377964467f, t, dyl[7]);
        }
        vfma(u17_11, a9.w, d17_62);
        { const float t = vdot(sx17_11, d17_62);
          dyl[6] = fmaf(-0.377964467f, t, dyl[6]);
          dyl[8] = fmaf(-0.327326834f, t, dyl[8]);
        }
        const float4 a11 = *reinterpret_cast<const float4*>(As + 44);
        vfma(u17_10, a11.x, d17_63);
        { const float t = vdot(sx17_10, d17_63);
          dyl[6] = fmaf(-0.597614288f, t, dyl[6]);
        }
        vfma(u17_12, a6.y, d17_59);
        { const float t = vdot(sx17_12, d17_59);
          dyl[8] = fmaf(0.267261237f, t, dyl[8]);
        }
        vfma(u17_12, a7.w, d17_60);
        { const float t = vdot(sx17_12, d17_60);
          dyl[7] = fmaf(-0.534522474f, t, dyl[7]);
        }
        vfma(u17_13, a9.x, d17_61);
        { const float t = vdot(sx17_13, d17_61);
          dyl[5] = fmaf(-0.377964467f, t, dyl[5]);
        }
        vfma(u17_12, a10.x, d17_62);
        { const float t = vdot(sx17_12, d17_62);
          dyl[5] = fmaf(0.534522474f, t, dyl[5]);
        }
        vfma(u17_11, a11.y, d17_63);
        { const float t = vdot(sx17_11, d17_63);
          dyl[7] = fmaf(0.327326834f, t, dyl[7]);
        }
        vfma(u17_13, a6.z, d17_59);
        { const float t = vdot(sx17_13, d17_59);
          dyl[7] = fmaf(-0.327326834f, t, dyl[7]);
        }
        vfma(u17_13, a8.x, d17_60);
        { const float t = vdot(sx17_13, d17_60);
          dyl[6] = fmaf(0.377964467f, t, dyl[6]);
          dyl[8] = fmaf(-0.327326834f, t, dyl[8]);
        }
        vfma(u17_14, a9.y, d17_61);
        { const float t = vdot(sx17_14, d17_61);
          dyl[4] = fmaf(-0.597614288f, t, dyl[4]);
        }
        vfma(u17_13, a10.y, d17_62);
        { const float t = vdot(sx17_13, d17_62);
          dyl[4] = fmaf(0.327326834f, t, dyl[4]);
        }
        vfma(u17_12, a11.z, d17_63);
        { const float t = vdot(sx17_12, d17_63);
          dyl[4] = fmaf(-0.267261237f, t, dyl[4]);
        }
        vfma(u17_14, a6.w, d17_59);
        { const float t = vdot(sx17_14, d17_59);
          dyl[6] = fmaf(0.597614288f, t, dyl[6]);
        }
        vfma(u17_15, a8.y, d17_60);
        { const float t = vdot(sx17_15, d17_60);
          dyl[8] = fmaf(-0.422577113f, t, dyl[8]);
        }
        vfma(u17_15, a10.z, d17_62);
        { const float t = vdot(sx17_15, d17_62);
          dyl[4] = fmaf(-0.422577113f, t, dyl[4]);
        }
        vfma(u17_13, a11.w, d17_63);
        { const float t = vdot(sx17_13, d17_63);
          dyl[5] = fmaf(0.327326834f, t, dyl[5]);
        }
        vfma(u17_15, a7.x, d17_59);
        { const float t = vdot(sx17_15, d17_59);
          dyl[7] = fmaf(0.422577113f, t, dyl[7]);
        }
        const float4 a12 = *reinterpret_cast<const float4*>(As + 48);
        vfma(u17_15, a12.x, d17_63);
        { const float t = vdot(sx17_15, d17_63);
          dyl[5] = fmaf(0.422577113f, t, dyl[5]);
        }
        EVec ds17 = vmul(x9, u17_9);
        vfma(ds17, x10, u17_10);
        vfma(ds17, x11, u17_11);
        vfma(ds17, x12, u17_12);
        vfma(ds17, x13, u17_13);
        vfma(ds17, x14, u17_14);
        vfma(ds17, x15, u17_15);
        if (gw) gw[17 * NQV] = ds17;
        vfma(dxp[9], s17, u17_9);
        vfma(dxp[10], s17, u17_10);
        vfma(dxp[11], s17, u17_11);
        vfma(dxp[12], s17, u17_12);
        vfma(dxp[13], s17, u17_13);
        vfma(dxp[14], s17, u17_14);
        vfma(dxp[15], s17, u17_15);
        dyl[9] = 0.f;
        dyl[10] = 0.f;
        dyl[11] = 0.f;
        dyl[12] = 0.f;
        dyl[13] = 0.f;
        dyl[14] = 0.f;
        dyl[15] = 0.f;
    }
};
}  // namespace
}  // namespace fast

extern const FastKernels kFast_q128_l2;
const FastKernels kFast_q128_l2 = {
    "128|0e+1o+2e+3o|2|0:0:0,1:1:0,2:2:0,0:1:1,1:0:1,1:2:1,2:1:1,3:2:1,1:1:1,2:2:1,0:2:2,1:1:2,2:0:2,2:2:2,3:1:2,1:2:2,2:1:2,3:2:2",
    &fast::fwd_scratch_bytes<fast::Sig_q128_l2>, &fast::bwd_scratch_bytes<fast::Sig_q128_l2>, &fast::launch_fwd<fast::Sig_q128_l2>, &fast::launch_bwd<fast::Sig_q128_l2>, &fast::launch_tp_fwd<fast::Sig_q128_l2>, &fast::launch_tp_bwd<fast::Sig_q128_l2>,
    nullptr, nullptr, nullptr, nullptr, 0};
}  // namespace e3j
