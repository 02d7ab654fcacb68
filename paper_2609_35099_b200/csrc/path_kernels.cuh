// Kernels for plans without generated ones, built from single coupling paths.
//
// A path (l1, l2) -> L with l <= 3 is one of 34 fixed tensors, so its pairs are unrolled with constant coefficients
// (fast/path_pairs.inc) whatever signature it belongs to; the plan only says which paths there are and where their
// rows lie.  A warp takes one path at a time (the switch below is warp-uniform) and keeps all rows of its result in
// registers while it walks its edges, so a path's input rows and weights are loaded once per edge instead of once
// per output row, and no coefficient record is ever fetched.
//
//   node sums  (forward; grad_x with the tensor transposed and the edges in sender order): one thread owns V channels
//              of one node and one block of rows, edges in list order; a node of many edges has several threads where the
//              nodes are few;
//   edge part  (grad_w, grad_sh): one thread owns V channels of one edge and walks all paths; grad_sh's channel sum
//              goes through shared memory in a fixed order.
//
// What bounds them: the latency of the row loads at 17 (backward) and 24 warps per SM (issue slots 50 and 41 % busy,
// DRAM 20 %), not arithmetic or bandwidth.  48x(0e+1o+2e), l <= 2, 35 050 edges: forward 243 -> 65 us, backward 823 ->
// 164 us against the table-driven kernels; float64, 64x(0e+1o), l <= 2, 10 176 edges, both passes: 715 -> 106 us.  Tried
// and slower: weights and ids two steps ahead in registers (spills, 378 against 284 us for both passes), each path's sum
// as a function of its own, grad_out rows of the next path in registers.
//
// Same sums as the table-driven kernels, in a fixed order, no atomics.  What stays on the table-driven ones: plans
// with l > 3, more than 128 V-channel units, and (float64) odd channel counts or pointers off 16 bytes.
#pragma once
#include "common.cuh"
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

// Tri<l1,l2,L>: sum    acc[m0] += w * (sum over the path's pairs of A(y)[m0,m1] in[m1])
//               sum_t  acc[m1] += w * (sum of A(y)[m0,m1] in[m0])
//               edge   dw += sum g[m0] A[m0,m1] x[m1],  dy[m2] += sum C (s x[m1]) . g[m0]
template <int l1, int l2, int L> struct Tri;

#define E3J_PB(o) { T z[V]; _Pragma("unroll") for (int c = 0; c < V; ++c) z[c] = T(0);
#define E3J_P1(r, i, a) axpy(z, T(a) * y[i], in[r]);
#define E3J_P2(r, i, a, j, b) axpy(z, fma(T(a), y[i], T(b) * y[j]), in[r]);
#define E3J_PE(o) axpy(acc[o], w, z); }
#define E3J_EB(o) { T z[V], sg[V]; _Pragma("unroll") for (int c = 0; c < V; ++c) { z[c] = T(0); sg[c] = s[c] * g[o][c]; }
#define E3J_E1(r, i, a) { axpy(z, T(a) * y[i], x[r]); dy[i] = fma(T(a), dot(x[r], sg), dy[i]); }
#define E3J_E2(r, i, a, j, b) { axpy(z, fma(T(a), y[i], T(b) * y[j]), x[r]); const T t_ = dot(x[r], sg); \
                                dy[i] = fma(T(a), t_, dy[i]); dy[j] = fma(T(b), t_, dy[j]); }
#define E3J_EE(o) axpy(dw, g[o], z); }
#define E3J_DEFINE_TRI(l1, l2, L)                                                                                    \
    template <> struct Tri<l1, l2, L> {                                                                              \
        static constexpr int kL1 = l1, kL2 = l2, kL = L;                                                             \
        template <class T, int V, int NI, int NO>                                                                    \
        __host__ __device__ static __forceinline__ void sum(const T* y, const T (&in)[NI][V], const T (&w)[V],       \
                                                            T (&acc)[NO][V]) {                                       \
            E3J_PATH_BY0_##l1##l2##L(E3J_PB, E3J_P1, E3J_P2, E3J_PE)                                                 \
        }                                                                                                            \
        template <class T, int V, int NI, int NO>                                                                    \
        __host__ __device__ static __forceinline__ void sum_t(const T* y, const T (&in)[NI][V], const T (&w)[V],     \
                                                              T (&acc)[NO][V]) {                                     \
            E3J_PATH_BY1_##l1##l2##L(E3J_PB, E3J_P1, E3J_P2, E3J_PE)                                                 \
        }                                                                                                            \
        template <class T, int V, int NX, int NG>                                                                    \
        __host__ __device__ static __forceinline__ void edge(const T* y, T* dy, const T (&x)[NX][V], const T (&s)[V],\
                                                             const T (&g)[NG][V], T (&dw)[V]) {                      \
            E3J_PATH_BY0_##l1##l2##L(E3J_EB, E3J_E1, E3J_E2, E3J_EE)                                                 \
        }                                                                                                            \
    };
E3J_PATH_TRIPLES(E3J_DEFINE_TRI)

template <class T> struct Args {
    int64_t n_nodes, n_edges;
    const T *x, *sh, *w, *g;     // g: grad_out
    const int32_t *senders, *receivers, *ptr, *perm, *n_real;
    T *out, *grad_w, *grad_sh;   // out: the node sums (forward out, backward grad_x)
    int d, dp, P, D, units;      // units: N_q / V
    int split_log2;              // a node has 2^split_log2 lanes; its own degree says to how many its edges are dealt
    unsigned group_blocks;
    unsigned node_blocks;        // backward: blocks below this one are node sums, the others edge tiles
};

// ---------------------------------------------------------------- staging
// In the edge part every lane copies its own rows into its own columns of a ring in shared memory (cp.async) two paths
// before it uses them: the loads in flight cost no registers, and no lane waits for another one (106 -> 89 us on the
// workload above).  The node sums keep plain loads: their copies are scattered over rows of many nodes, which the copy
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
            if constexpr (TR) Tr::template sum_t<T, V>(y[u], in[u], w[u], acc);
            else Tr::template sum<T, V>(y[u], in[u], w[u], acc);
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

// ---------------------------------------------------------------- edge part
template <class T, int V, int LM, bool IDENT>
__device__ __forceinline__ void edge_part(const PathTable& t, const Args<T>& a, const unsigned tile, unsigned char* smem) {
    const int slots = blockDim.x / a.units, slot = threadIdx.x / a.units, q = threadIdx.x - slot * a.units;
    const int64_t e = (int64_t)tile * slots + slot;
    const int64_t n_live = a.n_real ? min((int64_t)*a.n_real, a.n_edges) : a.n_edges;
    const bool mine = slot < slots && e < a.n_edges, live = mine && e < n_live;
    const int row = a.units * V;
    constexpr int NY = (LM + 1) * (LM + 1);
    T y[NY], dy[NY];
#pragma unroll
    for (int i = 0; i < NY; ++i) { dy[i] = T(0); y[i] = live && i < a.dp ? a.sh[(size_t)e * a.dp + i] : T(0); }
    if (live) {
        const int64_t from = IDENT ? e : (int64_t)a.senders[e], to = IDENT ? e : (int64_t)a.receivers[e];
        const T* xe = a.x + (size_t)from * a.d * row + q * V;
        const T* ge = a.g + (size_t)to * a.D * row + q * V;
        const T* we = a.w + (size_t)e * a.P * row + q * V;
        unsigned char* ring = smem + (threadIdx.x >> 5) * ring_bytes<LM>() + (threadIdx.x & 31) * 16;
        auto copy = [&](int p, int stage) {   // a path's weights and grad_out rows
            if (p < t.n_paths) {
                const PathRec rec = t.rec[p];
                unsigned char* at = ring + stage * stage_bytes<LM>();
                copy_async<16>(at, we + (size_t)rec.k * row);
                const T* gk = ge + (size_t)rec.out_off * row;
#pragma unroll
                for (int i = 0; i < 2 * LM + 1; ++i)
                    if (i < 2 * rec.L + 1) copy_async<16>(at + (1 + i) * 512, gk + (size_t)i * row);
            }
            copies_commit();
        };
        T x[2 * LM + 1][V];
#pragma unroll
        for (int i = 0; i < 2 * LM + 1; ++i)
#pragma unroll
            for (int c = 0; c < V; ++c) x[i][c] = T(0);
        int have = -1, stage = 0;
        copy(0, 0);
        copy(1, 1);
#pragma unroll 1
        for (int p = 0; p < t.n_paths; ++p) {
            const PathRec rec = t.rec[p];
            if (rec.x_off != have) {
                have = rec.x_off;
#pragma unroll
                for (int i = 0; i < 2 * LM + 1; ++i)
                    if (i < 2 * rec.l1 + 1) load_pack<T, V>(x[i], xe + (size_t)(rec.x_off + i) * row);
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
                    Tri<l1, l2, L>::template edge<T, V>(y + l2 * l2, dy + l2 * l2, x, s, g, dw); \
                } break;
                E3J_PATH_TRIPLES(E3J_CASE)
#undef E3J_CASE
            }
            if (a.grad_w) store_pack<T, V>(a.grad_w + ((size_t)e * a.P + rec.k) * row + q * V, dw);
        }
    } else if (mine && a.grad_w) {   // a padding edge: zero rows
        T z[V];
#pragma unroll
        for (int c = 0; c < V; ++c) z[c] = T(0);
        for (int k = 0; k < a.P; ++k) store_pack<T, V>(a.grad_w + ((size_t)e * a.P + k) * row + q * V, z);
    }
    if (!a.grad_sh) return;
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
// with them the blocks of an SM.  LM = 2, 48x(0e+1o+2e), 35 050 edges: the forward gains from more warps although values
// spill (99 / 95 / 71 us with 5 / 6 / 7 blocks), the backward does not (179 / 186 / 214 us).  LM = 3, geometric mean over
// six plans of 10 to 34 paths and 16 to 20 000 nodes: forward 1.08 / 1 / 0.93 with 3 / 4 / 5 blocks (16x(0e+1o+2e+3o), 35 000
// edges: 136 / 127 / 101 us), backward 0.97 / 1 / 1.16.  LM = 1, 96x0e: forward 1.04 / 1 / 1.02 and backward 1.06 / 1 /
// 1.06 with 6 / 8 / 10 blocks.
constexpr int kThreads = 128;
constexpr int fwd_blocks_per_sm(int lm) { return lm == 3 ? 5 : lm == 2 ? 7 : 8; }
constexpr int grad_x_blocks_per_sm(int lm) { return lm == 3 ? 4 : fwd_blocks_per_sm(lm); }
constexpr int bwd_blocks_per_sm(int lm) { return lm == 3 ? 4 : lm == 2 ? 5 : 8; }
template <int LM> constexpr int smem_bytes(int threads) { return threads / 32 * ring_bytes<LM>(); }

// TR: the forward's sums, or grad_x on its own.
template <class T, int V, int LM, bool TR, bool IDENT>
__global__ void __launch_bounds__(kThreads, TR ? grad_x_blocks_per_sm(LM) : fwd_blocks_per_sm(LM))
node_kernel(const __grid_constant__ PathTable t, const __grid_constant__ Args<T> a) {
    node_part<T, V, LM, TR, IDENT>(t, a, blockIdx.x);
}

// Edge tiles, and up to l = 2 the node sums of grad_x in the same launch (48x(0e+1o+2e), l <= 2: 180 us against 205 us
// one after the other).  With l = 3 the two parts' code together is too much for the instruction cache (16x(0e+1o+2e+3o),
// 35050 edges: 338 to 431 us against 264 us), so grad_x has its own launch; only where all blocks run at once do
// the parts share one, because there each is a chain of its paths' latencies (16 nodes of degree 5, the same signature:
// 74 -> 43 us; tensor product of 300 rows, 8x3o: 33 -> 18.5 us).
constexpr bool one_launch(int lm) { return lm < 3; }
template <class T, int V, int LM, bool IDENT, bool NODES>
__global__ void __launch_bounds__(kThreads, bwd_blocks_per_sm(LM))
bwd_kernel(const __grid_constant__ PathTable t, const __grid_constant__ Args<T> a) {
    extern __shared__ __align__(16) unsigned char smem[];
    static_assert((LM + 1) * (LM + 1) * 32 * (int)sizeof(T) <= ring_bytes<LM>(), "the partials take the rings' place");
    if constexpr (NODES) {
        if (blockIdx.x < a.node_blocks) {
            node_part<T, V, LM, true, IDENT>(t, a, blockIdx.x);
            return;
        }
    }
    edge_part<T, V, LM, IDENT>(t, a, blockIdx.x - a.node_blocks, smem);
}

}  // namespace path
}  // namespace e3j
