// Launchers of the per-path kernels (path_kernels.cuh), one translation unit per element type.
#pragma once
#include "path_kernels.cuh"

#include "path_launch.hpp"

namespace e3j {
namespace path {
namespace {

// Lanes per (node, unit, group): the edges of a node are walked by one lane while that fills the chip (`warps` per
// SM); smaller calls give a node up to 8 lanes, of which the kernel uses as many as get kLaneEdges edges each.  Not a
// function of the list's length: padding entries must not change the order of a sum.  The forward wants two lanes
// sooner (16x(0e+1o+2e+3o), 35 000 edges: 127 us with 32 warps, 151 with 16), the backward does not (the same signature,
// 3000 nodes of degree 1: 181 against 110 us; 48x(0e+1o+2e), 35 050 edges: 190 against 179).
// The sum of the shares is nothing but loads: two lanes until every SM has its 64 warps.
constexpr int kFwdWarps = 32, kBwdWarps = 16, kShareWarps = 64;
int split_of(int64_t n_nodes, int units, int groups, int warps) {
    int s = 0;
    while (s < 3 && (n_nodes * units * groups << s) < (int64_t)sm_count() * warps * 32) ++s;
    return s;
}

template <class T, int V> Args<T> args_of(const e3j_plan* plan, const Call<T>& c) {
    Args<T> a{};
    a.n_nodes = c.n_nodes; a.n_edges = c.n_edges; a.x = c.x; a.sh = c.sh; a.w = c.w; a.g = c.grad_out;
    a.senders = c.senders; a.receivers = c.receivers; a.n_real = c.n_real;
    a.d = plan->d; a.dp = plan->dp; a.P = plan->P; a.D = plan->D; a.units = plan->nq / V;
    return a;
}

inline int64_t node_blocks(int64_t n_nodes, int units, int split, int groups, int threads) {
    const int64_t items = n_nodes * units, per_block = threads >> split;
    return (items + per_block - 1) / per_block * groups;
}

template <class T, int V, int LM, bool IDENT> int fwd(const e3j_plan* plan, const Call<T>& c) {
    const bool pairs = !plan->path.shared_rows;
    const PathTable& t = pairs ? plan->path.by_pair : plan->path.by_output;
    Args<T> a = args_of<T, V>(plan, c);
    a.ptr = c.rowptr; a.out = c.out;
    a.split_log2 = IDENT ? 0 : split_of(c.n_nodes, a.units, t.n_groups, kFwdWarps);
    const int64_t blocks = node_blocks(c.n_nodes, a.units, a.split_log2, t.n_groups, kThreads);
    if (blocks >= (int64_t)1 << 31) return E3J_ERR_INVALID_ARG;
    a.group_blocks = (unsigned)(blocks / t.n_groups);
    if (pairs) {
        constexpr int few = few_pair_blocks_per_sm<T>(LM);
        constexpr int scalar_lx = LM > 1 ? 0 : LM;
        const auto kernel = blocks <= (int64_t)sm_count() * few ? pair_kernel<T, V, LM, IDENT, few>
                            : plan->path.largest_l1 == 0        ? pair_kernel<T, V, LM, IDENT, kScalarPairBlocks, scalar_lx>
                                                                : pair_kernel<T, V, LM, IDENT, pair_blocks_per_sm(LM)>;
        return launch_dependent(kernel, dim3((unsigned)blocks), dim3(kThreads), 0, c.stream, t, a);
    }
    node_kernel<T, V, LM, false, IDENT><<<(unsigned)blocks, kThreads, 0, c.stream>>>(t, a);
    return after_launch();
}

template <class T, int V, int LM, bool IDENT> int bwd(const e3j_plan* plan, const Call<T>& c) {
    const PathTable& t = plan->path.by_input;
    Args<T> a = args_of<T, V>(plan, c);
    a.ptr = c.colptr; a.perm = c.sender_perm; a.out = c.grad_x; a.grad_w = c.grad_w; a.grad_sh = c.grad_sh;
    const EdgeTable& et = sizeof(T) == 8 ? plan->path.edges_f64 : plan->path.edges_f32;
    const bool edges = (c.grad_w || c.grad_sh) && c.n_edges > 0;
    const bool from_shares = c.grad_x && (IDENT ? edges : c.shares && c.n_edges > 0);
    // block size: the multiple of 32 that leaves the fewest threads without an edge, the smaller of equals
    int threads = kThreads, best = 0;
    for (int b = 64; b <= kThreads; b += 32) {
        const int used = 1024 * (b / a.units * a.units) / b;
        if (used > best) { best = used; threads = b; }
    }
    const int64_t tiles = edges || from_shares ? (c.n_edges + threads / a.units - 1) / (threads / a.units) : 0;
    static_assert(smem_bytes<LM>(kThreads) <= 48 * 1024, "more would need the kernel's attribute set");
    if (c.grad_x && !from_shares) {
        a.split_log2 = IDENT ? 0 : split_of(c.n_nodes, a.units, t.n_groups, kBwdWarps);
        if constexpr (!IDENT) {   // (a tensor product whose edge gradients are wanted has grad_x from the edge part)
            const int64_t nodes = node_blocks(c.n_nodes, a.units, a.split_log2, t.n_groups, threads);
            if (tiles > 0 && (one_launch(LM) || nodes + tiles <= (int64_t)sm_count() * joint_blocks_per_sm(LM))) {
                if (nodes + tiles >= (int64_t)1 << 31) return E3J_ERR_INVALID_ARG;
                a.group_blocks = (unsigned)(nodes / t.n_groups);
                a.node_blocks = (unsigned)nodes;
                joint_kernel<T, V, LM><<<(unsigned)(nodes + tiles), threads, smem_bytes<LM>(threads), c.stream>>>(t, et, a);
                return after_launch();
            }
        }
        const int64_t nodes = node_blocks(c.n_nodes, a.units, a.split_log2, t.n_groups, kThreads);
        if (nodes >= (int64_t)1 << 31) return E3J_ERR_INVALID_ARG;
        a.group_blocks = (unsigned)(nodes / t.n_groups);
        node_kernel<T, V, LM, true, IDENT><<<(unsigned)nodes, kThreads, 0, c.stream>>>(t, a);
        if (int s = after_launch()) return s;
    }
    if (tiles > 0) {
        if (tiles >= (int64_t)1 << 31) return E3J_ERR_INVALID_ARG;
        a.dx = !from_shares ? nullptr : IDENT ? c.grad_x : c.shares;
        constexpr int all = edge_blocks_per_sm<T>(LM);
        const bool at_once = tiles * threads <= (int64_t)sm_count() * all * kThreads;
        const auto kernel = !from_shares     ? edge_kernel<T, V, LM, IDENT, Want::kEdges, edges_alone_blocks_per_sm<T>(LM)>
                            : edges || IDENT ? edge_kernel<T, V, LM, IDENT, Want::kAll, all>
                            : at_once        ? edge_kernel<T, V, LM, false, Want::kX, all>
                                             : edge_kernel<T, V, LM, false, Want::kX, only_x_blocks_per_sm<T>(LM)>;
        if (int s = launch_dependent(kernel, dim3((unsigned)tiles), dim3(threads), smem_bytes<LM>(threads), c.stream, et, a)) return s;
    }
    if (!from_shares || IDENT) return E3J_OK;
    a.dx = c.shares;
    a.split_log2 = split_of(c.n_nodes, a.d * a.units, 1, kShareWarps);
    const int64_t blocks = node_blocks(c.n_nodes, a.d * a.units, a.split_log2, 1, kThreads);
    if (blocks >= (int64_t)1 << 31) return E3J_ERR_INVALID_ARG;
    return launch_dependent(share_sum_kernel<T, V>, dim3((unsigned)blocks), dim3(kThreads), 0, c.stream, a);
}

}  // namespace

#define E3J_BY_LARGEST_L(f, T, V, IDENT)                  \
    switch (plan->path.largest_l) {                       \
        case 1: return f<T, V, 1, IDENT>(plan, c);        \
        case 2: return f<T, V, 2, IDENT>(plan, c);        \
        default: return f<T, V, 3, IDENT>(plan, c);       \
    }

}  // namespace path
}  // namespace e3j
