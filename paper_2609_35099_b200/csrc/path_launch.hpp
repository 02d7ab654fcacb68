// Internal: entry to the per-path kernels for plans without generated ones (path_kernels.cuh).
#pragma once
#include "common.cuh"

namespace e3j {
namespace path {

template <class T> struct Call {
    int64_t n_nodes, n_edges;
    const T *x, *sh, *w, *grad_out;
    const int32_t *senders, *receivers, *rowptr, *sender_perm, *colptr, *n_real;
    T *out, *grad_x, *grad_sh, *grad_w;
    T* shares;   // backward: room for [n_edges, d, N_q] shares of grad_x, or null: grad_x is summed from the edges' inputs
    cudaStream_t stream;
};

// All l <= 3, channels in whole groups of `vec` and at most 128 of them (a thread owns one group of an edge, a block
// at least one edge).
bool covers(const e3j_plan* plan, int vec);
// Does the backward sum grad_x from per-edge shares where it has room for them?  With scalar inputs alone it does not: a
// node sum there reads two to four weights and a few rows per edge, in the launch of the edge tiles.  The line was drawn by one case
// (96x0e, l <= 1, 300 nodes x 200 edges: 53 us against 68) and is not the best one: over 54 calls of six such plans the shares take
// 0.78 of the node sums' time, 0.85 in float64; from a third for 4 nodes of degree 400 to 1.3 for 16 nodes of degree 5 and, in float64
// at l <= 3, 1.27 for 75 000 edges (445 against 567 us).
inline bool uses_shares(const e3j_plan* plan) { return plan->path.largest_l1 > 0; }
int conv_fwd(const e3j_plan* plan, const Call<float>& c, bool ident);   // four channels per thread
int conv_bwd(const e3j_plan* plan, const Call<float>& c, bool ident);
int conv_fwd(const e3j_plan* plan, const Call<double>& c);              // two; arrays on 16-byte boundaries
int conv_bwd(const e3j_plan* plan, const Call<double>& c);

}  // namespace path
}  // namespace e3j
