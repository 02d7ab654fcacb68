// Kernels for plans without generated ones, built from single coupling paths.
//
// A path (l1, l2) -> L with l <= 3 is one of 34 fixed tensors, so its pairs are unrolled with constant coefficients
// (fast/path_pairs.inc) whatever signature it belongs to; the plan only says which paths there are and where their
// rows lie.  A warp takes one path at a time (the switch below is warp-uniform) and keeps all rows of its result in
// registers while it walks its edges, so a path's input rows and weights are loaded once per edge instead of once
// per output row, and no coefficient record is ever fetched.
//
//   forward    one thread owns V channels of one node and the output blocks of one (input block, l2), edges in list
//              order; a node of many edges has several threads where the nodes are few;
//   backward   edge part: one thread owns V channels of one edge and walks all paths by input block, for grad_w, grad_sh
//              (its channel sum goes through shared memory in a fixed order) and the edge's share of grad_x, which a second
//              kernel adds up over the sender-sorted list;
//   node sums by single output blocks: the forward of plans whose paths share output rows, and grad_x (tensor transposed,
//              edges in sender order) where the workspace has no room for the shares or where every input is scalar.
//
// What bounds them, 48x(0e+1o+2e), l <= 2, 35 050 edges: the edge part its instructions (90 us, 60 % of the issue slots, half
// of them multiply-adds), the forward the latency of its row loads at 24 warps per SM (50 us, 45 % of the issue slots), the
// sum of the shares its loads (16 us).  Both passes 218 -> 157 us against one thread per output block with grad_x from the
// edges' inputs (every path's input rows and harmonics loaded again, the weights read twice in the backward); float64,
// 64x(0e+1o), l <= 2, 10 176 edges: 106 -> 77 us.  Tried and slower: a block's tiles one after the other with the copies
// running on from tile to tile and the input rows among them (fewer warps fit: backward 106 -> 145 us); weights and ids two
// steps ahead in registers (spills), each path's sum as a function of its own, grad_out rows of the next path in registers.
//
// Same sums as the table-driven kernels, in a fixed order, no atomics.  What stays on the table-driven ones: plans
// with l > 3, more than 128 V-channel units, and (float64) odd channel counts or pointers off 16 bytes.
#pragma once
#include "common.cuh"
#include "fast/fast_common.cuh"
#include "fast/path_pairs.inc"
#include "path_table.hpp"

namespace e3j {
namespace path {

template <class T, int V> struct alignas(sizeof(T) * V) Pack { T v[V]; };

template <class T, int V>
__host__ __device__ __forceinline__ void load_pack(T (&dst)[V], const T* src) {
    const Pack<T, V> p = *reinterpret_cast<const Pack<T, V>*>(src);
#pragma unroll
    for (int c = 0; c < V; ++c) dst[c] = p.v[c];
}
template <class T, int V>
__host__ __device__ __forceinline__ void store_pack(T* dst, const T (&src)[V]) {
    Pack<T, V> p;
#pragma unroll
    for (int c = 0; c < V; ++c) p.v[c] = src[c];
    *reinterpret_cast<Pack<T, V>*>(dst) = p;
}
template <class T, int V, int N>
__host__ __device__ __forceinline__ void clear(T (&z)[N][V]) {
#pragma unroll
    for (int o = 0; o < N; ++o)
#pragma unroll
        for (int c = 0; c < V; ++c) z[o][c] = T(0);
}
template <class T, int V>
__host__ __device__ __forceinline__ void axpy(T (&z)[V], const T a, const T (&x)[V]) {
#pragma unroll
    for (int c = 0; c < V; ++c) z[c] = fma(a, x[c], z[c]);
}
template <class T, int V>
__host__ __device__ __forceinline__ void axpy(T (&z)[V], const T (&a)[V], const T (&x)[V]) {
#pragma unroll
    for (int c = 0; c < V; ++c) z[c] = fma(a[c], x[c], z[c]);
}
template <class T, int V>
__host__ __device__ __forceinline__ T dot(const T (&a)[V], const T (&b)[V]) {
    T s = a[0] * b[0];
#pragma unroll
    for (int c = 1; c < V; ++c) s = fma(a[c], b[c], s);
    return s;
}

// Tri<l1,l2,L>: sum    acc[AT + m0] += w * (sum over the path's pairs of A(y)[m0,m1] in[m1])
//               sum_t  acc[m1] += w * (sum of A(y)[m0,m1] in[m0])
//               edge   u = sum of A[m0,m1] g[m0];  dw += x[m1] u,  dx[m1] += s u,  dy[m2] += C (s x[m1]) . g[m0]
template <int l1, int l2, int L> struct Tri;

#define E3J_PB(o) { T z[V]; _Pragma("unroll") for (int c = 0; c < V; ++c) z[c] = T(0);
#define E3J_P1(r, i, a) axpy(z, T(a) * y[i], in[r]);
#define E3J_P2(r, i, a, j, b) axpy(z, fma(T(a), y[i], T(b) * y[j]), in[r]);
#define E3J_PE(o) axpy(acc[AT + o], w, z); }
#define E3J_EB(o) { T u[V], sx[V]; _Pragma("unroll") for (int c = 0; c < V; ++c) { u[c] = T(0); sx[c] = s[c] * x[o][c]; }
#define E3J_E1(r, i, a) { axpy(u, T(a) * y[i], g[r]); dy[i] = fma(T(a), dot(sx, g[r]), dy[i]); }
#define E3J_E2(r, i, a, j, b) { axpy(u, fma(T(a), y[i], T(b) * y[j]), g[r]); const T t_ = dot(sx, g[r]); \
                                dy[i] = fma(T(a), t_, dy[i]); dy[j] = fma(T(b), t_, dy[j]); }
#define E3J_EE(o) axpy(dw, x[o], u); if constexpr (DX) axpy(dx[o], s, u); }
#define E3J_DEFINE_TRI(l1, l2, L)                                                                                    \
    template <> struct Tri<l1, l2, L> {                                                                              \
        static constexpr int kL1 = l1, kL2 = l2, kL = L;                                                             \
        template <int AT, class T, int V, int NI, int NO>                                                            \
        __host__ __device__ static __forceinline__ void sum(const T* y, const T (&in)[NI][V], const T (&w)[V],       \
                                                            T (&acc)[NO][V]) {                                       \
            E3J_PATH_BY0_##l1##l2##L(E3J_PB, E3J_P1, E3J_P2, E3J_PE)                                                 \
        }                                                                                                            \
        template <int AT, class T, int V, int NI, int NO>                                                            \
        __host__ __device__ static __forceinline__ void sum_t(const T* y, const T (&in)[NI][V], const T (&w)[V],     \
                                                              T (&acc)[NO][V]) {                                     \
            E3J_PATH_BY1_##l1##l2##L(E3J_PB, E3J_P1, E3J_P2, E3J_PE)                                                 \
        }                                                                                                            \
        template <bool DX, class T, int V, int NX, int NG>                                                           \
        __host__ __device__ static __forceinline__ void edge(const T* y, T* dy, const T (&x)[NX][V], const T (&s)[V],\
                                                             const T (&g)[NG][V], T (&dw)[V], T (&dx)[NX][V]) {      \
            E3J_PATH_BY1_##l1##l2##L(E3J_EB, E3J_E1, E3J_E2, E3J_EE)                                                 \
        }                                                                                                            \
    };
E3J_PATH_TRIPLES(E3J_DEFINE_TRI)

template <class T> struct Args {
    int64_t n_nodes, n_edges;
    const T *x, *sh, *w, *g;     // g: grad_out
    const int32_t *senders, *receivers, *ptr, *perm, *n_real;
    T *out, *grad_w, *grad_sh;   // out: the node sums (forward out, backward grad_x)
    T* dx;                       // each edge's share of grad_x, [n_edges, d, N_q] (null: not wanted)
    int d, dp, P, D, units;      // units: N_q / V
    int split_log2;              // a node has 2^split_log2 lanes; its own degree says to how many its edges are dealt
    unsigned group_blocks;
    unsigned node_blocks;        // joint launch: blocks below this one are node sums, the others edge tiles
};

// ---------------------------------------------------------------- staging
// In the edge part every lane copies its own rows into its own columns of a ring in shared memory (cp.async) two paths
// before it uses them: the loads in flight cost no registers, and no lane waits for another one (106 -> 89 us for grad_w and
// grad_sh of the workload above).  The node sums keep plain loads: their copies are scattered over rows of many nodes, which the copy
// path takes at half the rate (99 -> 148 us).
constexpr int kStages = 3;
template <int BYTES> __device__ __forceinline__ void copy_async(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;"
                 :: "r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT> __device__ __forceinline__ void copies_wait() {
    asm volatile("cp.async.wait_group %0;" :: "n"(LEFT) : "memory");
}
// A stage of one warp: up to 2 LM + 2 rows of one Pack per lane.
template <int LM> constexpr int stage_bytes() { return (2 * LM + 2) * 512; }
template <int LM> constexpr int ring_bytes() { return kStages * stage_bytes<LM>(); }

// ---------------------------------------------------------------- node sums
// One path's share of a node's rows, summed over the lane's edges (every step-th one) and added to acc.
template <class Tr, class T, int V, bool TR, bool IDENT>
__device__ __forceinline__ void walk_path(const Args<T>& a, const PathRec rec, const unsigned j0, const unsigned j1,
                                         const int step, const int row, const int q,
                                         T (&acc)[TR ? 2 * Tr::kL1 + 1 : 2 * Tr::kL + 1][V]) {
    constexpr int NI = TR ? 2 * Tr::kL + 1 : 2 * Tr::kL1 + 1, NO = TR ? 2 * Tr::kL1 + 1 : 2 * Tr::kL + 1;
    constexpr int NY = 2 * Tr::kL2 + 1;
    constexpr int U = NI <= 3 ? 2 : 1;   // edges in flight: with three input rows or fewer two fit, with w and y of each
    const T* in_base = (TR ? a.g + (size_t)rec.out_off * row : a.x + (size_t)rec.x_off * row) + q * V;
    const T* w_base = a.w + (size_t)rec.k * row + q * V;
    const size_t in_stride = (size_t)(TR ? a.D : a.d) * row, w_stride = (size_t)a.P * row;
    // the ids of an edge are fetched one step ahead of its rows; past the end: the last step's first edge again
    int e[U], b[U];
    auto ids = [&](unsigned j) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned jc = j + u * step < j1 ? j + u * step : j;
            e[u] = TR && !IDENT ? a.perm[jc] : (int)jc;
            b[u] = IDENT ? e[u] : TR ? a.receivers[e[u]] : a.senders[e[u]];
        }
    };
    if (j0 < j1) ids(j0);
#pragma unroll 1
    for (unsigned j = j0; j < j1; j += U * step) {
        T in[U][NI][V], y[U][NY], w[U][V];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            load_pack<T, V>(w[u], w_base + (size_t)e[u] * w_stride);
#pragma unroll
            for (int i = 0; i < NI; ++i) load_pack<T, V>(in[u][i], in_base + (size_t)b[u] * in_stride + i * row);
#pragma unroll
            for (int i = 0; i < NY; ++i) y[u][i] = a.sh[(size_t)e[u] * a.dp + rec.y_off + i];
        }
        if (j + U * step < j1) ids(j + U * step);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (j + u * step >= j1) break;
            if constexpr (TR) Tr::template sum_t<0, T, V>(y[u], in[u], w[u], acc);
            else Tr::template sum<0, T, V>(y[u], in[u], w[u], acc);
        }
    }
}
// The forward's groups: added up over the lanes that share the node and stored by the first of them (added to the rows for
// the second and later paths of a collapsed block).
template <class Tr, class T, int V, bool TR, bool IDENT>
__device__ __forceinline__ void sum_path(const Args<T>& a, const PathRec rec, const unsigned j0, const unsigned j1,
                                         const int step, const int used, const int row, const int q, T* dst, const bool first) {
    constexpr int NO = TR ? 2 * Tr::kL1 + 1 : 2 * Tr::kL + 1;
    T acc[NO][V];
    clear(acc);
    walk_path<Tr, T, V, TR, IDENT>(a, rec, j0, j1, step, row, q, acc);
#pragma unroll 1
    for (int off = 32 >> a.split_log2; off < (32 >> a.split_log2) * used; off <<= 1) {
#pragma unroll
        for (int o = 0; o < NO; ++o)
#pragma unroll
            for (int c = 0; c < V; ++c) acc[o][c] += __shfl_xor_sync(0xffffffffu, acc[o][c], off);
    }
    if (!dst) return;
#pragma unroll
    for (int o = 0; o < NO; ++o) {
        if (!first) {
            T have[V];
            load_pack<T, V>(have, dst + (size_t)o * row);
#pragma unroll
            for (int c = 0; c < V; ++c) acc[o][c] += have[c];
        }
        store_pack<T, V>(dst + (size_t)o * row, acc[o]);
    }
}

// The backward's groups have several paths each: their sums, each taken by itself, are added in registers, then over the
// lanes, and stored once.
template <int LO, class T, int V, int LM, bool IDENT>
__device__ __forceinline__ void node_group(const PathTable& t, const Args<T>& a, const int p0, const int p1, const unsigned j0,
                                           const unsigned j1, const int step, const int used, const int row, const int q, T* dst) {
    constexpr int NO = 2 * LO + 1;
    T tot[NO][V];
    clear(tot);
#pragma unroll 1
    for (int p = p0; p < p1; ++p) {
        const PathRec rec = t.rec[p];
        int row_p = row, step_p = step;
        asm volatile("" : "+r"(row_p), "+r"(step_p));
        switch (rec.id) {
#define E3J_CASE(l1, l2, L) \
            case tri_id(l1, l2, L): \
                if constexpr (l1 == LO && l2 <= LM && L <= LM) { \
                    if constexpr (IDENT) {   /* one edge: nothing to sum apart */ \
                        walk_path<Tri<l1, l2, L>, T, V, true, IDENT>(a, rec, j0, j1, step_p, row_p, q, tot); \
                    } else { \
                        T acc[NO][V]; \
                        clear(acc); \
                        walk_path<Tri<l1, l2, L>, T, V, true, IDENT>(a, rec, j0, j1, step_p, row_p, q, acc); \
                        _Pragma("unroll") for (int o = 0; o < NO; ++o) \
                            _Pragma("unroll") for (int c = 0; c < V; ++c) tot[o][c] += acc[o][c]; \
                    } \
                } \
                break;
            E3J_PATH_TRIPLES(E3J_CASE)
#undef E3J_CASE
        }
    }
#pragma unroll 1
    for (int off = 32 >> a.split_log2; off < (32 >> a.split_log2) * used; off <<= 1) {
#pragma unroll
        for (int o = 0; o < NO; ++o)
#pragma unroll
            for (int c = 0; c < V; ++c) tot[o][c] += __shfl_xor_sync(0xffffffffu, tot[o][c], off);
    }
    if (!dst) return;
#pragma unroll
    for (int o = 0; o < NO; ++o) store_pack<T, V>(dst + (size_t)o * row, tot[o]);
}

constexpr int kLaneEdges = 4;   // a lane's edges at least, where a node's edges are dealt to several

template <class T, int V, int LM, bool TR, bool IDENT>
__device__ __forceinline__ void node_part(const PathTable& t, const Args<T>& a, const unsigned block) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int per_warp = 32 >> a.split_log2, part = lane >> (5 - a.split_log2);
    // From l = 2 on a group's blocks follow one another, so that an SM runs few different paths at a time (instruction
    // cache; 20 000 nodes of degree 3, 16x(0e+1o+2e+3o): grad_x 589 -> 328 us), the last groups, which have the highest l,
    // first.  With l <= 1 the few paths fit, and the groups of one node run side by side, which read the same rows
    // (49 157 rows of a tensor product, 384x1o: 223 against 252 us).
    unsigned turn, at;
    if constexpr (LM >= 2) { turn = block / a.group_blocks; at = block - turn * a.group_blocks; }
    else { at = block / (unsigned)t.n_groups; turn = block - at * (unsigned)t.n_groups; }
    const int grp = t.n_groups - 1 - (int)turn;
    const int64_t item = ((int64_t)at * warps + warp) * per_warp + (lane & (per_warp - 1));
    const int64_t node = item / a.units;
    const int q = (int)(item - node * a.units), row = a.units * V;
    unsigned j0 = 0, j1 = 0;   // edge counts are below 2^31, so a step past the end does not wrap
    int step = 1;
    T* dst = nullptr;
    const int p0 = t.start[grp], p1 = t.start[grp + 1];
    if (node < a.n_nodes) {
        j0 = IDENT ? (unsigned)node : (unsigned)a.ptr[node];
        j1 = IDENT ? (unsigned)node + 1 : (unsigned)a.ptr[node + 1];
        while (step < 1 << a.split_log2 && j1 - j0 >= 2u * kLaneEdges * step) step *= 2;
        j0 = part < step ? j0 + part : j1;
        if (part == 0)
            dst = a.out + ((size_t)node * (TR ? a.d : a.D) + (TR ? t.rec[p0].x_off : t.rec[p0].out_off)) * row + q * V;
    }
    const int used = IDENT ? 1 : __reduce_max_sync(0xffffffffu, step);
    if constexpr (TR) {
        if (t.rec[p0].id == kNoPath) {   // zero rows
            T z[V];
#pragma unroll
            for (int c = 0; c < V; ++c) z[c] = T(0);
            if (dst)
                for (int o = 0; o < 2 * t.rec[p0].l1 + 1; ++o) store_pack<T, V>(dst + (size_t)o * row, z);
            return;
        }
        switch (t.rec[p0].l1) {
            case 0: node_group<0, T, V, LM, IDENT>(t, a, p0, p1, j0, j1, step, used, row, q, dst); break;
            case 1: node_group<1, T, V, LM, IDENT>(t, a, p0, p1, j0, j1, step, used, row, q, dst); break;
            case 2: if constexpr (LM >= 2) node_group<2, T, V, LM, IDENT>(t, a, p0, p1, j0, j1, step, used, row, q, dst); break;
            case 3: if constexpr (LM >= 3) node_group<3, T, V, LM, IDENT>(t, a, p0, p1, j0, j1, step, used, row, q, dst); break;
        }
        return;
    }
#pragma unroll 1
    for (int p = p0; p < p1; ++p) {
        const PathRec rec = t.rec[p];
        int row_p = row, step_p = step;
        asm volatile("" : "+r"(row_p), "+r"(step_p));   // keeps every case's address arithmetic inside the case
        switch (rec.id) {
#define E3J_CASE(l1, l2, L) \
            case tri_id(l1, l2, L): \
                if constexpr (l1 <= LM && l2 <= LM && L <= LM) \
                    sum_path<Tri<l1, l2, L>, T, V, TR, IDENT>(a, rec, j0, j1, step_p, used, row_p, q, dst, p == p0); \
                break;
            E3J_PATH_TRIPLES(E3J_CASE)
#undef E3J_CASE
        }
    }
}

// The forward by (input block, l2): a thread walks its edges once for all paths of a group, so the sender's rows and the
// harmonics are loaded once for up to three output blocks and the work between two loads is that of all of them.  Where
// several paths share an output block (collapsed plans) the groups above take it.
template <class Tr, int AT, class T, int V, int NI, int NO>
__device__ __forceinline__ void add_path(const bool has, const T* y, const T (&x)[NI][V], const T (&w)[V], T (&acc)[NO][V]) {
    if (has) Tr::template sum<AT, T, V>(y, x, w, acc);
}
template <int l1, int l2, int LA, int LB, class T, int V, bool IDENT>
__device__ __forceinline__ void pair_group(const PathTable& t, const Args<T>& a, const int p0, const int p1, const unsigned j0,
                                           const unsigned j1, const int step, const int used, const int row, const int q, T* dst) {
    constexpr int NI = 2 * l1 + 1, NY = 2 * l2 + 1, NL = LB - LA + 1, ROWS = (LB + 1) * (LB + 1) - LA * LA;
    static_assert(NL <= 3, "paths to L = 3 have groups of their own where a pair has others");
    bool has[NL];   // the output filter may have dropped some
    int k[NL], out_off[NL];
    for (int i = 0, p = p0; i < NL; ++i) {
        has[i] = p < p1 && t.rec[p].L == LA + i;
        k[i] = has[i] ? t.rec[p].k * row : 0;
        out_off[i] = has[i] ? t.rec[p].out_off * row : 0;
        p += has[i];
    }
    const PathRec rec = t.rec[p0];
    const T* x_base = a.x + (size_t)rec.x_off * row + q * V;
    const T* w_base = a.w + q * V;
    const size_t x_stride = (size_t)a.d * row, w_stride = (size_t)a.P * row;
    T acc[ROWS][V];
    clear(acc);
    int b = j0 < j1 ? (IDENT ? (int)j0 : a.senders[j0]) : 0;
#pragma unroll 1
    for (unsigned j = j0; j < j1; j += step) {
        T x[NI][V], y[NY], w[NL][V];
        const T* we = w_base + (size_t)j * w_stride;
        const T* xe = x_base + (size_t)b * x_stride;
#pragma unroll
        for (int i = 0; i < NL; ++i)
            if (has[i]) load_pack<T, V>(w[i], we + k[i]);
#pragma unroll
        for (int i = 0; i < NI; ++i) load_pack<T, V>(x[i], xe + (size_t)i * row);
#pragma unroll
        for (int i = 0; i < NY; ++i) y[i] = a.sh[(size_t)j * a.dp + rec.y_off + i];
        if (!IDENT && j + step < j1) b = a.senders[j + step];
        add_path<Tri<l1, l2, LA>, 0, T, V>(has[0], y, x, w[0], acc);
        if constexpr (NL > 1) add_path<Tri<l1, l2, LA + 1>, (LA + 1) * (LA + 1) - LA * LA, T, V>(has[1], y, x, w[1], acc);
        if constexpr (NL > 2) add_path<Tri<l1, l2, LA + 2>, (LA + 2) * (LA + 2) - LA * LA, T, V>(has[2], y, x, w[2], acc);
    }
#pragma unroll 1
    for (int off = 32 >> a.split_log2; off < (32 >> a.split_log2) * used; off <<= 1) {
#pragma unroll
        for (int o = 0; o < ROWS; ++o)
#pragma unroll
            for (int c = 0; c < V; ++c) acc[o][c] += __shfl_xor_sync(0xffffffffu, acc[o][c], off);
    }
    if (!dst) return;
#pragma unroll
    for (int i = 0; i < NL; ++i) {
        const int L = LA + i;
        if (!has[i]) continue;
#pragma unroll
        for (int o = 0; o < 2 * L + 1; ++o) store_pack<T, V>(dst + out_off[i] + (size_t)o * row, acc[L * L - LA * LA + o]);
    }
}

template <class T, int V, int LM, int LX, bool IDENT>   // LX: the largest l of the inputs
__device__ __forceinline__ void pair_part(const PathTable& t, const Args<T>& a, const unsigned block) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int per_warp = 32 >> a.split_log2, part = lane >> (5 - a.split_log2);
    unsigned turn, at;   // in the order of node_part, for the same reasons (48x(0e+1o+2e), 35 050 edges: 61 -> 55 us)
    if constexpr (LM >= 2) { turn = block / a.group_blocks; at = block - turn * a.group_blocks; }
    else { at = block / (unsigned)t.n_groups; turn = block - at * (unsigned)t.n_groups; }
    const int grp = t.n_groups - 1 - (int)turn;
    const int64_t item = ((int64_t)at * warps + warp) * per_warp + (lane & (per_warp - 1));
    const int64_t node = item / a.units;
    const int q = (int)(item - node * a.units), row = a.units * V;
    unsigned j0 = 0, j1 = 0;
    int step = 1;
    T* dst = nullptr;
    const int p0 = t.start[grp], p1 = t.start[grp + 1];
    if (node < a.n_nodes) {
        j0 = IDENT ? (unsigned)node : (unsigned)a.ptr[node];
        j1 = IDENT ? (unsigned)node + 1 : (unsigned)a.ptr[node + 1];
        while (step < 1 << a.split_log2 && j1 - j0 >= 2u * kLaneEdges * step) step *= 2;
        j0 = part < step ? j0 + part : j1;
        if (part == 0) dst = a.out + (size_t)node * a.D * row + q * V;
    }
    const int used = IDENT ? 1 : __reduce_max_sync(0xffffffffu, step);
    const PathRec rec = t.rec[p0];
    switch (rec.id >> 2) {
#define E3J_CASE(l1, l2) \
        case l1 * 4 + l2: { \
            constexpr int lo = l1 > l2 ? l1 - l2 : l2 - l1, hi = l1 + l2 < LM ? l1 + l2 : LM; \
            if constexpr (l1 <= LX && l2 <= LM && lo <= hi) { \
                constexpr bool split = hi == 3 && lo < 3; \
                if constexpr (split) { \
                    if (rec.L == 3) { pair_group<l1, l2, 3, 3, T, V, IDENT>(t, a, p0, p1, j0, j1, step, used, row, q, dst); break; } \
                } \
                pair_group<l1, l2, lo, split ? 2 : hi, T, V, IDENT>(t, a, p0, p1, j0, j1, step, used, row, q, dst); \
            } \
        } break;
        E3J_CASE(0, 0) E3J_CASE(0, 1) E3J_CASE(0, 2) E3J_CASE(0, 3) E3J_CASE(1, 0) E3J_CASE(1, 1) E3J_CASE(1, 2) E3J_CASE(1, 3)
        E3J_CASE(2, 0) E3J_CASE(2, 1) E3J_CASE(2, 2) E3J_CASE(2, 3) E3J_CASE(3, 0) E3J_CASE(3, 1) E3J_CASE(3, 2) E3J_CASE(3, 3)
#undef E3J_CASE
    }
}

// ---------------------------------------------------------------- edge part
// All three gradients, the shares of grad_x alone (to the same bits), or grad_w and grad_sh alone (16x(0e+1o+2e+3o), 35 050
// edges: grad_w 100 us with the shares formed all the same, 85 without; 48x(0e+1o+2e), l <= 2: 74 and 64 us).
enum class Want { kAll, kX, kEdges };
template <class T, int V, int LM, bool IDENT, Want WANT>
__device__ __forceinline__ void edge_part(const EdgeTable& t, const Args<T>& a, const unsigned tile, unsigned char* smem) {
    const int slots = blockDim.x / a.units, slot = threadIdx.x / a.units, q = threadIdx.x - slot * a.units;
    const int64_t e = (int64_t)tile * slots + slot;
    const int64_t n_live = a.n_real ? min((int64_t)*a.n_real, a.n_edges) : a.n_edges;
    const bool mine = slot < slots && e < a.n_edges, live = mine && e < n_live;
    constexpr int NY = (LM + 1) * (LM + 1), ROWS = 2 * LM + 1;
    constexpr bool ONLY_X = WANT == Want::kX, DX = WANT != Want::kEdges;
    const int row = a.units * V;
    const uint32_t row_bytes = (uint32_t)(row * sizeof(T)), unit = (uint32_t)(q * V * sizeof(T));
    T y[NY], dy[NY];
#pragma unroll
    for (int i = 0; i < NY; ++i) { dy[i] = T(0); y[i] = live && i < a.dp ? a.sh[(size_t)e * a.dp + i] : T(0); }
    if (live) {
        const int64_t from = IDENT ? e : (int64_t)a.senders[e], to = IDENT ? e : (int64_t)a.receivers[e];
        const char* xe = reinterpret_cast<const char*>(a.x) + (size_t)from * a.d * row_bytes + unit;
        const char* ge = reinterpret_cast<const char*>(a.g) + (size_t)to * a.D * row_bytes + unit;
        const char* we = reinterpret_cast<const char*>(a.w) + (size_t)e * a.P * row_bytes + unit;
        char* const gw = reinterpret_cast<char*>(a.grad_w) + (size_t)e * a.P * row_bytes + unit;
        char* const gx = reinterpret_cast<char*>(a.dx) + (size_t)e * a.d * row_bytes + unit;
        unsigned char* ring = smem + (threadIdx.x >> 5) * ring_bytes<LM>() + (threadIdx.x & 31) * 16;
        auto copy = [&](int p, int stage) {   // a path's weights and grad_out rows
            if (p < t.n_paths) {
                const EdgeRec r = t.rec[p];
                unsigned char* at = ring + stage * stage_bytes<LM>();
                copy_async<16>(at, we + r.w);
                const char* gk = ge + r.g;
#pragma unroll
                for (int i = 0; i < ROWS; ++i) {
                    if (i < r.n_g) copy_async<16>(at + (1 + i) * 512, gk);
                    gk += row_bytes;
                }
            }
            copies_commit();
        };
        T x[ROWS][V], dx[ROWS][V];   // the input block of the paths at hand, and this edge's share of its gradient
        clear(x);
        clear(dx);
        int x_rows = 0, stage = 0;
        uint32_t x_at = 0;
        auto put_dx = [&] {
            if (!DX || !a.dx) return;
            char* at = gx + x_at;
#pragma unroll
            for (int i = 0; i < ROWS; ++i) {
                if (i < x_rows) store_pack<T, V>(reinterpret_cast<T*>(at), dx[i]);
                at += row_bytes;
            }
        };
        copy(0, 0);
        copy(1, 1);
#pragma unroll 1
        for (int p = 0; p < t.n_paths; ++p) {
            const EdgeRec rec = t.rec[p];
            if (rec.n_x) {
                put_dx();
                clear(dx);
                x_rows = rec.n_x;
                x_at = rec.x;
                const char* at = xe + rec.x;
#pragma unroll
                for (int i = 0; i < ROWS; ++i) {
                    if (!ONLY_X && i < x_rows) load_pack<T, V>(x[i], reinterpret_cast<const T*>(at));
                    at += row_bytes;
                }
            }
            copies_wait<1>();
            copy(p + 2, stage == 0 ? 2 : stage - 1);
            const unsigned char* at = ring + stage * stage_bytes<LM>();
            stage = stage == 2 ? 0 : stage + 1;
            T s[V], dw[V];
            load_pack<T, V>(s, reinterpret_cast<const T*>(at));
#pragma unroll
            for (int c = 0; c < V; ++c) dw[c] = T(0);
            switch (rec.id) {
#define E3J_CASE(l1, l2, L) \
                case tri_id(l1, l2, L): if constexpr (l1 <= LM && l2 <= LM && L <= LM) { \
                    T g[2 * L + 1][V]; \
                    _Pragma("unroll") for (int i = 0; i < 2 * L + 1; ++i) \
                        load_pack<T, V>(g[i], reinterpret_cast<const T*>(at + (1 + i) * 512)); \
                    if constexpr (ONLY_X) Tri<l1, l2, L>::template sum_t<0, T, V>(y + l2 * l2, g, s, dx); \
                    else Tri<l1, l2, L>::template edge<DX, T, V>(y + l2 * l2, dy + l2 * l2, x, s, g, dw, dx); \
                } break;
                E3J_PATH_TRIPLES(E3J_CASE)
#undef E3J_CASE
            }
            if (!ONLY_X && a.grad_w) store_pack<T, V>(reinterpret_cast<T*>(gw + rec.w), dw);
        }
        put_dx();
        if (DX && a.dx) {
            T z[V];
#pragma unroll
            for (int c = 0; c < V; ++c) z[c] = T(0);
            for (int k = t.n_paths; k < t.n_recs; ++k)   // input rows that no path reads
                for (uint32_t i = 0; i < t.rec[k].n_x; ++i) store_pack<T, V>(reinterpret_cast<T*>(gx + t.rec[k].x + i * row_bytes), z);
        }
    } else if (mine && a.grad_w) {   // a padding edge: zero rows
        T z[V];
#pragma unroll
        for (int c = 0; c < V; ++c) z[c] = T(0);
        for (int k = 0; k < a.P; ++k) store_pack<T, V>(a.grad_w + ((size_t)e * a.P + k) * row + q * V, z);
    }
    if (ONLY_X || !a.grad_sh) return;
    copies_wait<0>();
    __syncthreads();   // the rings are free: the partials take their place
    T* part = reinterpret_cast<T*>(smem);
    // channel sum: 2^lanes_log2 lanes per (edge, component), eight where there are as many partials, add every eighth
    // partial each, then a fixed tree over them.  With few units there are many sums of few terms: eight lanes for each
    // took 128 rounds with one unit (backward of a tensor product, 4x(0e+1o+2e+3o), 300 rows: 84 -> 49 us)
#pragma unroll
    for (int i = 0; i < NY; ++i)
        if (i < a.dp) part[i * blockDim.x + threadIdx.x] = dy[i];
    __syncthreads();
    const int lanes_log2 = a.units > 4 ? 3 : a.units > 2 ? 2 : a.units - 1, lanes = 1 << lanes_log2;
    const int sub = threadIdx.x & (lanes - 1), n_out = slots * a.dp, per_pass = blockDim.x >> lanes_log2;
    for (int o0 = 0; o0 < n_out; o0 += per_pass) {
        const int o = o0 + (threadIdx.x >> lanes_log2);
        const int sl = o / a.dp, i = o - sl * a.dp;
        T sum = T(0);
        if (o < n_out)
            for (int u = sub; u < a.units; u += lanes) sum += part[i * blockDim.x + sl * a.units + u];
#pragma unroll 1
        for (int off = lanes >> 1; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
        const int64_t eo = (int64_t)tile * slots + sl;
        if (sub == 0 && o < n_out && eo < a.n_edges) a.grad_sh[(size_t)eo * a.dp + i] = sum;
    }
}

// LM: the plan's largest l.  It sets the registers of a thread (an edge's input rows, harmonics and grad_out rows) and
// with them the blocks of an SM.  Geometric means over some sixty calls of eleven plans (8 to 256 channels, 16 to 20 000
// nodes), blocks per SM of LM = 1 / 2 / 3.  Forward by pairs, against one thread per output block: 0.88 with 6 / 5 / 4, 0.85
// with 8 / 6 / 5 although values spill, 0.88 with 10 / 7 / 6.  Edge part, float32: more blocks spill (backward 0.77 with 6 / 4 / 3,
// 1.00 with 8 / 5 / 4), fewer help only 80x(0e+1o+2e), l <= 3 (0.68 -> 0.61 with 2); float64 fits one block less (64x(0e+1o): l <= 2
// 1.02 -> 0.86, l <= 3 0.72 -> 0.63).  Node sums: measured as the only kernels (LM = 2 forward 99 / 95 / 71 us with 5 / 6 / 7).
constexpr int kThreads = 128;
constexpr int fwd_blocks_per_sm(int lm) { return lm == 3 ? 5 : lm == 2 ? 7 : 8; }
constexpr int grad_x_blocks_per_sm(int lm) { return lm == 3 ? 4 : fwd_blocks_per_sm(lm); }
constexpr int joint_blocks_per_sm(int lm) { return lm == 3 ? 4 : lm == 2 ? 5 : 8; }
constexpr int pair_blocks_per_sm(int lm) { return lm == 3 ? 5 : lm == 2 ? 6 : 8; }
// Where the forward's blocks all run at once with fewer of them per SM, a block is a chain of its edges' latencies, and the
// spilled values lengthen it: the same kernel with more registers (8 / 4 / 3, float64 8 / 3 / 3).  Six blocks at l = 2 and five
// at l = 3 against it, 4 nodes of degree 400: 48x(0e+1o+2e), l <= 2, 51 -> 34 us, float64 68 -> 37; 16x(0e+1o+2e+3o), l <= 3, 50 ->
// 39, float64 64 -> 45.  64 nodes of degree 20, the first: 9.2 -> 6.3.  Large launches want the blocks: 1500 x 50, the first,
// 143 us against 185 with four; 6000 x 20, the other, 249 against 341 with three.
// Scalar inputs alone, from l = 2 on: the kernel without the other inputs' cases fits eight blocks per SM in its registers.  96x0e,
// 75 000 edges, with the six and five blocks of the whole kernel, with this one, and by output blocks: l <= 2 56 / 46 / 48 us, float64 113 /
// 96 / 93; l <= 3 90 / 65 / 88, float64 167 / 123 / 157.  Where all blocks run at once it is up to 1.6 times as long as the one above.
constexpr int kScalarPairBlocks = 8;
template <class T> constexpr int few_pair_blocks_per_sm(int lm) { return lm == 3 || (lm == 2 && sizeof(T) == 8) ? 3 : lm == 2 ? 4 : 8; }
template <class T> constexpr int edge_blocks_per_sm(int lm) {
    return sizeof(T) == 8 ? (lm == 3 ? 2 : lm == 2 ? 3 : 5) : (lm == 3 ? 3 : lm == 2 ? 4 : 6);
}
// grad_w and grad_sh alone.  In float64 the eight and four blocks of l = 1 and 3 spill (1100 bytes at l = 3); one less: geometric
// means over 18 and 74 calls 0.84 / 0.66 for grad_w, 0.92 / 0.80 for grad_sh (120x1o, l <= 1, 120 000 edges: grad_w 295 -> 195 us).
// A second one less at l = 1 gives grad_w two per cent more and takes up to seven from a grad_sh.  At l = 2 one less makes grad_w
// 0.85, and the grad_sh of scalar inputs up to 1.25 where 740 blocks ran at once and 592 do not.
template <class T> constexpr int edges_alone_blocks_per_sm(int lm) { return joint_blocks_per_sm(lm) - (sizeof(T) == 8 && lm != 2 ? 1 : 0); }
// grad_x alone in float64: where its blocks do not all run at once, one more per SM.  64x(0e+1o), l <= 3, 5000 edges 37 -> 27 us;
// 128x(0e+1o), 6000 edges 81 -> 61; in launches that do it costs up to a quarter (4x(0e+1o), l <= 3, 5000 edges 12.4 -> 15.5).
template <class T> constexpr int only_x_blocks_per_sm(int lm) { return edge_blocks_per_sm<T>(lm) + (sizeof(T) == 8 ? 1 : 0); }
template <int LM> constexpr int smem_bytes(int threads) { return threads / 32 * ring_bytes<LM>(); }

// TR: the forward's sums, or grad_x on its own.
template <class T, int V, int LM, bool TR, bool IDENT>
__global__ void __launch_bounds__(kThreads, TR ? grad_x_blocks_per_sm(LM) : fwd_blocks_per_sm(LM))
node_kernel(const __grid_constant__ PathTable t, const __grid_constant__ Args<T> a) {
    node_part<T, V, LM, TR, IDENT>(t, a, blockIdx.x);
}

template <class T, int V, int LM, bool IDENT, int BLOCKS, int LX = LM>
__global__ void __launch_bounds__(kThreads, BLOCKS)
pair_kernel(const __grid_constant__ PathTable t, const __grid_constant__ Args<T> a) {
    fast::grid_dependency_wait();
    pair_part<T, V, LM, LX, IDENT>(t, a, blockIdx.x);
}

template <class T, int V, int LM, bool IDENT, Want WANT, int BLOCKS>
__global__ void __launch_bounds__(kThreads, BLOCKS)
edge_kernel(const __grid_constant__ EdgeTable et, const __grid_constant__ Args<T> a) {
    extern __shared__ __align__(16) unsigned char smem[];
    static_assert((LM + 1) * (LM + 1) * 32 * (int)sizeof(T) <= ring_bytes<LM>(), "the partials take the rings' place");
    fast::grid_dependency_wait();
    edge_part<T, V, LM, IDENT, WANT>(et, a, blockIdx.x, smem);
}

// Edge tiles, and up to l = 2 the node sums of grad_x in the same launch.  With l = 3 the two parts' code together is too
// much for the instruction cache (16x(0e+1o+2e+3o), 35050 edges: 338 to 431 us against 264 us), so grad_x has its own
// launch; only where all blocks run at once do the parts share one, because there each is a chain of its paths' latencies.
constexpr bool one_launch(int lm) { return lm < 3; }
template <class T, int V, int LM>
__global__ void __launch_bounds__(kThreads, joint_blocks_per_sm(LM))
joint_kernel(const __grid_constant__ PathTable t, const __grid_constant__ EdgeTable et, const __grid_constant__ Args<T> a) {
    extern __shared__ __align__(16) unsigned char smem[];
    if (blockIdx.x < a.node_blocks) {
        node_part<T, V, LM, true, false>(t, a, blockIdx.x);
        return;
    }
    edge_part<T, V, LM, false, Want::kEdges>(et, a, blockIdx.x - a.node_blocks, smem);
}

// grad_x from the edges' shares: one 16-byte unit of a node's row to 2^split_log2 lanes, which take every so manieth
// edge of the sender-sorted list each, eight loads in flight.
constexpr int kShareLoads = 8;
template <class T, int V>
__global__ void __launch_bounds__(kThreads)
share_sum_kernel(const __grid_constant__ Args<T> a) {
    const int lane = threadIdx.x & 31;
    const int per_warp = 32 >> a.split_log2, part = lane >> (5 - a.split_log2);
    const int64_t item = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * per_warp + (lane & (per_warp - 1));
    const int row_units = a.d * a.units;
    const int64_t node = item / row_units;
    const int i = (int)(item - node * row_units);
    unsigned j0 = 0, j1 = 0;
    int step = 1;
    if (node < a.n_nodes) {
        j0 = (unsigned)a.ptr[node];
        j1 = (unsigned)a.ptr[node + 1];
        while (step < 1 << a.split_log2 && j1 - j0 >= 2u * kLaneEdges * step) step *= 2;
        j0 = part < step ? j0 + part : j1;
    }
    const int used = __reduce_max_sync(0xffffffffu, step);
    fast::grid_dependency_wait();
    fast::grid_dependency_trigger();
    T acc[V];
#pragma unroll
    for (int c = 0; c < V; ++c) acc[c] = T(0);
    const T* from = a.dx + (size_t)i * V;
#pragma unroll 1
    for (unsigned j = j0; j < j1; j += kShareLoads * step) {
        T v[kShareLoads][V];
        clear(v);
#pragma unroll
        for (int u = 0; u < kShareLoads; ++u)
            if (j + u * step < j1) load_pack<T, V>(v[u], from + (size_t)a.perm[j + u * step] * row_units * V);
#pragma unroll
        for (int u = 0; u < kShareLoads; ++u)
#pragma unroll
            for (int c = 0; c < V; ++c) acc[c] += v[u][c];
    }
#pragma unroll 1
    for (int off = 32 >> a.split_log2; off < (32 >> a.split_log2) * used; off <<= 1)
#pragma unroll
        for (int c = 0; c < V; ++c) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], off);
    if (node < a.n_nodes && part == 0) store_pack<T, V>(a.out + (size_t)item * V, acc);
}

}  // namespace path
}  // namespace e3j
