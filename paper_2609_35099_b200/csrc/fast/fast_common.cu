// Kernels shared by all signature-specialised entries.
#include "../common.cuh"
#include "fast_common.cuh"

namespace e3j {
namespace fast {

__global__ void fwd_fixup_kernel(int n_cta, int row_f4, const float4* __restrict__ partial,
                                 const int32_t* __restrict__ part_recv, float4* __restrict__ out) {
    grid_dependency_wait();
    grid_dependency_trigger();
    const int c = blockIdx.x;
    const int b = part_recv[2 * c + 1];  // a row whose first piece is this CTA's tail
    if (b < 0) return;
    int last = c;
    while (last + 1 < n_cta && part_recv[2 * (last + 1)] == b) ++last;
    for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < row_f4; i += gridDim.y * blockDim.x) {
        float4 sum = partial[(size_t)(2 * c + 1) * row_f4 + i];
        for (int c2 = c + 1; c2 <= last; ++c2) {
            const float4 v = partial[(size_t)(2 * c2) * row_f4 + i];
            sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
        }
        out[(size_t)b * row_f4 + i] = sum;
    }
}

// One warp, one barrier with one expected arrival that never comes, no copy in flight: the wait runs out after
// `limit` polls, records the time-out in *status and returns false; result[0] = what the wait returned,
// result[1] = the CTA's abort flag afterwards.  Nothing here can hang: the loop is bounded by `limit`.
__global__ void bounded_wait_selftest_kernel(uint32_t limit, int32_t* status, int32_t* result) {
    __shared__ uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) { mbar_init(&bar, 1); abort_flag = 0; mbar_fence_init(); }
    __syncthreads();
    const bool ok = mbar_wait_limit(&bar, 0, &abort_flag, status, limit);
    __syncthreads();
    if (threadIdx.x == 0) { result[0] = ok ? 1 : 0; result[1] = abort_flag; }
}

namespace {
__device__ __forceinline__ void zero_padding_rows(const ZeroPadding& z, int64_t block, int64_t n_blocks) {
    const int64_t first = min((int64_t)*z.n_real, z.n_edges);
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int64_t e = first + block; e < z.n_edges; e += n_blocks) {
        if (z.grad_w)
            for (int i = threadIdx.x; i < z.w_row_f4; i += blockDim.x) z.grad_w[(size_t)e * z.w_row_f4 + i] = zero;
        if (z.grad_sh)
            for (int i = threadIdx.x; i < z.sh_row; i += blockDim.x) z.grad_sh[(size_t)e * z.sh_row + i] = 0.f;
    }
}
}  // namespace

__global__ void bwd_zero_padding_kernel(ZeroPadding z) { zero_padding_rows(z, blockIdx.x, gridDim.x); }

// The most runs a sender's edges are dealt to: as many as the senders leave room for on the chip, in blocks of 1024.
static int most_runs(int64_t n_nodes, int row_f4) {
    int runs = 1;
    while (runs < 8 && n_nodes * row_f4 * runs < (int64_t)sm_count() * 2048 && 2 * runs * row_f4 <= 1024) runs *= 2;
    return runs;
}
constexpr int kRunEdges = 8;   // a run's edges at most, up to that many runs: one batch of loads

// 32 registers: with more, the 16 blocks of 128 threads that hide the row loads' latency do not fit an SM (36: 217 ->
// 227 us for the backward of 20 000 nodes and 40 000 edges, 128x(0e+1o)).
__global__ void __launch_bounds__(1024, 2)
bwd_dx_reduce_kernel(int64_t n_nodes, int row_f4, int max_runs, const float4* __restrict__ dx_edge,
                                     const int32_t* __restrict__ sender_perm, const int32_t* __restrict__ colptr,
                                     float4* __restrict__ grad_x, ZeroPadding pad) {
    extern __shared__ float4 part[];   // [max_runs][row_f4] where max_runs > 1
    if (blockIdx.x >= n_nodes) {   // padding rows: not the sweep's, which itself started after all that came before it
        zero_padding_rows(pad, blockIdx.x - n_nodes, gridDim.x - n_nodes);
        return;
    }
    const int64_t a = blockIdx.x;
    const int groups = blockDim.x / row_f4, grp = threadIdx.x / row_f4, i = threadIdx.x - grp * row_f4;
    const int b0 = colptr[a], n = colptr[a + 1] - b0;
    int runs = 1;
    while (runs < max_runs && n > kRunEdges * runs) runs *= 2;
    const int per = (n + runs - 1) / runs;
    grid_dependency_wait();
    grid_dependency_trigger();
    float4 acc;
    for (int r = grp; r < runs; r += groups) {
        const int j1 = b0 + min(n, (r + 1) * per);
        acc = make_float4(0.f, 0.f, 0.f, 0.f);
        // eight independent loads in flight; the additions stay in edge order
        for (int j = b0 + r * per; j < j1; j += 8) {
            float4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                v[u] = j + u < j1 ? dx_edge[(size_t)sender_perm[j + u] * row_f4 + i] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 8; ++u) { acc.x += v[u].x; acc.y += v[u].y; acc.z += v[u].z; acc.w += v[u].w; }
        }
        if (runs > 1) part[r * row_f4 + i] = acc;
    }
    if (runs > 1) __syncthreads();
    if (grp > 0) return;
    if (runs > 1) {
        acc = part[i];
        for (int r = 1; r < runs; ++r) {
            const float4 v = part[r * row_f4 + i];
            acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
        }
    }
    grad_x[(size_t)a * row_f4 + i] = acc;
}

int launch_dx_reduce(int64_t n_nodes, int64_t n_edges, int row_f4, const float* dx_edge, const int32_t* sender_perm,
                     const int32_t* colptr, float* grad_x, const ZeroPadding& pad, cudaStream_t st) {
    const int runs = most_runs(n_nodes, row_f4);
    int groups = 1;   // as many as the average sender has runs
    while (groups < runs && n_edges > n_nodes * groups * kRunEdges) groups *= 2;
    const int64_t blocks = n_nodes + (pad.n_real ? sm_count() * 4 : 0);
    return launch_dependent(bwd_dx_reduce_kernel, dim3((unsigned)blocks), dim3(row_f4 * groups),
                            sizeof(float4) * (runs > 1 ? runs : 0) * row_f4, st, n_nodes, row_f4, runs,
                            reinterpret_cast<const float4*>(dx_edge), sender_perm, colptr, reinterpret_cast<float4*>(grad_x), pad);
}

__global__ void bwd_rows_reduce_kernel(int64_t n_nodes, int row_f4, const float4* __restrict__ dx_rows,
                                       const int32_t* __restrict__ row_ptr, float4* __restrict__ grad_x) {
    grid_dependency_wait();
    for (int64_t a = blockIdx.x; a < n_nodes; a += gridDim.x) {
        const int j0 = row_ptr[a], j1 = row_ptr[a + 1];
        for (int i = threadIdx.x; i < row_f4; i += blockDim.x) {
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            int j = j0;
            for (; j + 8 <= j1; j += 8) {   // eight independent loads in flight; the additions stay in row order
                float4 v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = dx_rows[(size_t)(j + u) * row_f4 + i];
#pragma unroll
                for (int u = 0; u < 8; ++u) { acc.x += v[u].x; acc.y += v[u].y; acc.z += v[u].z; acc.w += v[u].w; }
            }
            for (; j < j1; ++j) {
                const float4 v = dx_rows[(size_t)j * row_f4 + i];
                acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
            }
            grad_x[(size_t)a * row_f4 + i] = acc;
        }
    }
}

}  // namespace fast
}  // namespace e3j

