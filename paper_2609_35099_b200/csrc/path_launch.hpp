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
    cudaStream_t stream;
};

// All l <= 3, channels in whole groups of `vec` and at most 128 of them (a thread owns one group of an edge, a block
// at least one edge).
bool covers(const e3j_plan* plan, int vec);
int conv_fwd(const e3j_plan* plan, const Call<float>& c, bool ident);   // four channels per thread
int conv_bwd(const e3j_plan* plan, const Call<float>& c, bool ident);
int conv_fwd(const e3j_plan* plan, const Call<double>& c);              // two; arrays on 16-byte boundaries
int conv_bwd(const e3j_plan* plan, const Call<double>& c);

}  // namespace path
}  // namespace e3j
