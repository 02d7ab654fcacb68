// Graph preparation on the device: receiver CSR pointers and the sender-sorted edge
// permutation used by the backward ("message passing on the transposed graph").
// Integer work only; integer atomics are used to claim slots, and every bucket is
// sorted afterwards so the result does not depend on the order they were claimed in.
#include <algorithm>

#include "common.cuh"
#include "fast/fast_common.cuh"

namespace e3j {
namespace {

// rowptr[b] = first edge whose receiver is >= b.  All n_nodes + 1 entries are written with values in [0, n_edges]
// whatever the ids are.  Called by whole warps, tid and n_threads counted over all of them.
// Up to kFillNodes nodes: every edge that opens new receivers writes their entries (a warp writes one edge's entries
// together), what lies behind the last edge is dealt to all threads.  One pass of coalesced loads: a binary search per
// receiver takes 18 dependent ones (80 000 edges, 1536 receivers: 12.0 against 7.5 us as a call of its own).
// Beyond, the search per receiver: a run of receivers without edges is written by one warp in the first form, 32 at a
// step, however long it is (100 edges, half of them at the last node: 65 536 nodes 10.3 us against 11.9, 200 000 nodes
// 25.1 against 11.9, 10 million 1099 against 92), and with as many receivers as that the search is not slower either
// (100 000 nodes, 4.77 million edges: 14.4 against 12.0 us).
constexpr int64_t kFillNodes = 65536;
__device__ __forceinline__ void fill_rowptr(int64_t n_nodes, int64_t n_edges, const int32_t* __restrict__ receivers,
                                            int32_t* __restrict__ rowptr, int64_t tid, int64_t n_threads) {
    if (n_nodes > kFillNodes) {
        for (int64_t b = tid; b <= n_nodes; b += n_threads) {
            int64_t lo = 0, hi = n_edges;
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (receivers[mid] < b) lo = mid + 1; else hi = mid;
            }
            rowptr[b] = (int32_t)lo;
        }
        return;
    }
    const int lane = threadIdx.x & 31;
    const int32_t n = (int32_t)n_nodes;
    for (int64_t e0 = tid - lane; e0 < n_edges; e0 += n_threads) {
        const int64_t e = e0 + lane;
        int32_t lo = 0, hi = -1;
        if (e < n_edges) {
            hi = min(receivers[e], n);
            lo = e > 0 ? max(min(receivers[e - 1], n) + 1, 0) : 0;
        }
        for (unsigned open = __ballot_sync(0xffffffffu, hi >= lo); open; open &= open - 1) {
            const int src = __ffs(open) - 1;
            const int32_t first = __shfl_sync(0xffffffffu, lo, src), last = __shfl_sync(0xffffffffu, hi, src);
            for (int32_t b = first + lane; b <= last; b += 32) rowptr[b] = (int32_t)(e0 + src);
        }
    }
    const int64_t rest = n_edges > 0 ? max(min(receivers[n_edges - 1], n) + 1, 0) : 0;
    for (int64_t b = rest + tid; b <= n_nodes; b += n_threads) rowptr[b] = (int32_t)n_edges;
}

__global__ void rowptr_kernel(int64_t n_nodes, int64_t n_edges, const int32_t* __restrict__ receivers,
                              int32_t* __restrict__ rowptr) {
    fill_rowptr(n_nodes, n_edges, receivers, rowptr, blockIdx.x * (int64_t)blockDim.x + threadIdx.x,
                (int64_t)gridDim.x * blockDim.x);
}

// `pad_recv`: when not null, edges whose receiver id is >= n_nodes are padding and are left out.
__global__ void count_senders_kernel(int64_t n_nodes, int64_t n_edges, const int32_t* __restrict__ senders,
                                     const int32_t* __restrict__ pad_recv, int32_t* __restrict__ colptr) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n_edges;
         e += (int64_t)gridDim.x * blockDim.x) {
        if (pad_recv && pad_recv[e] >= n_nodes) continue;
        atomicAdd(&colptr[senders[e]], 1);
    }
}

// In-place exclusive scan of v[0..n) by one block; v[n] receives the total.
__global__ void __launch_bounds__(1024) exclusive_scan_kernel(int64_t n, int32_t* __restrict__ v) {
    __shared__ int32_t warp_sums[32];
    __shared__ int32_t carry_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry_s = 0;
    __syncthreads();
    for (int64_t base = 0; base < n; base += blockDim.x) {
        const int64_t i = base + threadIdx.x;
        const int32_t mine = (i < n) ? v[i] : 0;
        int32_t incl = mine;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int32_t up = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += up;
        }
        if (lane == 31) warp_sums[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            int32_t ws = warp_sums[lane];
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int32_t up = __shfl_up_sync(0xffffffffu, ws, off);
                if (lane >= off) ws += up;
            }
            warp_sums[lane] = ws;  // inclusive over warps
        }
        __syncthreads();
        const int32_t carry = carry_s;
        const int32_t before = carry + (warp ? warp_sums[warp - 1] : 0) + incl - mine;
        if (i < n) v[i] = before;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry_s = before + mine;
        __syncthreads();
    }
    if (threadIdx.x == 0) v[n] = carry_s;
}

// Claims a slot for every edge; afterwards colptr[a] is the END of bucket a.
__global__ void fill_kernel(int64_t n_nodes, int64_t n_edges, const int32_t* __restrict__ senders,
                            const int32_t* __restrict__ pad_recv, int32_t* __restrict__ colptr,
                            int32_t* __restrict__ perm) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n_edges;
         e += (int64_t)gridDim.x * blockDim.x) {
        if (pad_recv && pad_recv[e] >= n_nodes) continue;
        const int32_t pos = atomicAdd(&colptr[senders[e]], 1);
        perm[pos] = (int32_t)e;
    }
}

__device__ inline void sift_down(int32_t* v, int64_t root, int64_t n) {
    while (true) {
        int64_t child = 2 * root + 1;
        if (child >= n) return;
        if (child + 1 < n && v[child + 1] > v[child]) ++child;
        if (v[root] >= v[child]) return;
        const int32_t tmp = v[root]; v[root] = v[child]; v[child] = tmp;
        root = child;
    }
}

// Sorts every bucket ascending by edge id.  colptr holds bucket ENDS here.
// One warp per bucket.  Edge ids are distinct, so an element's place is the number of smaller ones: buckets
// of up to kRankMax entries are staged in shared memory and every lane counts the ranks of its elements;
// a longer bucket (a hub sender) is heap-sorted in place by one lane.
constexpr int kRankMax = 1024;
constexpr int kSortWarps = 4;

// One warp sorts the bucket v[0..n), with `stage` (MAX entries of shared memory) to itself.
template <int MAX>
__device__ __forceinline__ void sort_bucket(int32_t* v, int64_t n, int32_t* stage) {
    const int lane = threadIdx.x & 31;
    if (n <= 1) return;
    if (n <= MAX) {
        for (int i = lane; i < n; i += 32) stage[i] = v[i];
        __syncwarp();
        for (int i = lane; i < n; i += 32) {
            const int32_t key = stage[i];
            int rank = 0;
            for (int j = 0; j < n; ++j) rank += stage[j] < key;
            v[rank] = key;
        }
        __syncwarp();
    } else if (lane == 0) {
        for (int64_t i = n / 2 - 1; i >= 0; --i) sift_down(v, i, n);
        for (int64_t end = n - 1; end > 0; --end) {
            const int32_t tmp = v[0]; v[0] = v[end]; v[end] = tmp;
            sift_down(v, 0, end);
        }
    }
}

__global__ void __launch_bounds__(32 * kSortWarps)
sort_buckets_kernel(int64_t n_nodes, const int32_t* __restrict__ colptr, int32_t* __restrict__ perm) {
    __shared__ int32_t stage[kSortWarps][kRankMax];
    const int warp = threadIdx.x >> 5;
    for (int64_t a = (int64_t)blockIdx.x * kSortWarps + warp; a < n_nodes; a += (int64_t)gridDim.x * kSortWarps) {
        const int64_t begin = a ? colptr[a - 1] : 0;
        sort_bucket<kRankMax>(perm + begin, colptr[a] - begin, stage[warp]);
    }
}

// colptr[a] (end of bucket a) -> colptr[a+1]; colptr[0] = 0.  One block, top down.
__global__ void __launch_bounds__(1024) shift_up_kernel(int64_t n_nodes, int32_t* __restrict__ colptr) {
    for (int64_t hi = n_nodes; hi > 0; hi -= blockDim.x) {
        const int64_t i = hi - 1 - threadIdx.x;  // source index
        int32_t val = 0;
        if (i >= 0) val = colptr[i];
        __syncthreads();
        if (i >= 0) colptr[i + 1] = val;
        __syncthreads();
    }
    if (threadIdx.x == 0) colptr[0] = 0;
}

__global__ void validate_kernel(int64_t n_nodes, int64_t n_edges, const int32_t* __restrict__ senders,
                                const int32_t* __restrict__ receivers, int32_t* __restrict__ status) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n_edges;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t s = senders[e], r = receivers[e];
        bool bad = s < 0 || s >= n_nodes || r < 0 || r >= n_nodes;
        if (e > 0 && receivers[e - 1] > r) bad = true;
        if (bad) *status = E3J_ERR_GRAPH;  // every writer stores the same value
    }
}

// The whole preparation of a list of up to kOneLaunchEdges edges in one launch without any exchange between blocks:
// every block reads all sender ids, collects the edges of its own run of nodes in shared memory and counts those of the
// nodes before it, which gives it its place in the permutation.  The six kernels it stands for run 3 to 5 us each at
// these sizes, nearly all of it launch and first-load latency (12 288 edges, 192 nodes: 25 -> 8.7 us; 81 408 edges,
// 1536 nodes: 31 -> 14 us).  Tried and slower: a cluster of 16 blocks with the counters in each other's shared memory
// (13.5 / 32 us).  Its time is that of reading the ids through one SM
// (4 bytes x edges at some 64 bytes a cycle) and grows with the list: as calls, 24.6 against 40 us at 160 900 edges, 28.7
// against 43 at 196 608, to where it was measured; the kernels above take 51 us at 200 000.
constexpr int kOneThreads = 1024, kOneWarps = kOneThreads / 32;
constexpr int64_t kOneLaunchEdges = 196608;
constexpr int kOneBlocks = 128, kOneNodes = 2048;   // blocks at most, nodes per block at most
constexpr int kOneCap = 8192;                       // collected edges of a block at most; more: the ids are read again

struct OneSmem {
    int32_t edge[kOneCap], node[kOneCap];   // as collected: edge id; local node << 13 | place in its bucket
    int32_t key[kOneCap], of[kOneCap];      // by bucket: edge id, local node
    int32_t start[kOneNodes + 1];           // edges sent, then first place of the bucket
    int32_t warp_sum[kOneWarps];
    int32_t collected, before;              // the block's edges; edges of the nodes before the block's
};
static_assert(kOneCap <= 1 << 13 && kOneNodes <= 1 << 18, "a collected edge's node and place share a word");

// f(edge, sender) for every real edge, 16-byte loads where the ids start on a 16-byte boundary.
template <class F>
__device__ __forceinline__ void for_senders(int64_t n_nodes, int64_t n_edges, const int32_t* __restrict__ senders,
                                            const int32_t* __restrict__ pad_recv, F f) {
    auto real = [&](int64_t e) { return !(pad_recv && pad_recv[e] >= n_nodes); };
    int64_t done = 0;
    if (((uintptr_t)senders & 15u) == 0) {
        const int4* s4 = reinterpret_cast<const int4*>(senders);
        done = n_edges / 4 * 4;
        for (int64_t i = threadIdx.x; i < done / 4; i += 4 * kOneThreads) {
            int4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i + u * kOneThreads < done / 4) v[u] = s4[i + u * kOneThreads];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t e = 4 * (i + u * kOneThreads);
                if (e >= done) break;
                if (real(e)) f(e, v[u].x);
                if (real(e + 1)) f(e + 1, v[u].y);
                if (real(e + 2)) f(e + 2, v[u].z);
                if (real(e + 3)) f(e + 3, v[u].w);
            }
        }
    }
    for (int64_t e = done + threadIdx.x; e < n_edges; e += kOneThreads)
        if (real(e)) f(e, senders[e]);
}

__global__ void __launch_bounds__(kOneThreads)
prepare_one_kernel(int64_t n_nodes, int64_t n_edges, const int32_t* __restrict__ senders,
                   const int32_t* __restrict__ receivers, const int32_t* __restrict__ pad_recv,
                   int32_t* __restrict__ rowptr, int32_t* __restrict__ colptr, int32_t* __restrict__ perm, int per_block) {
    extern __shared__ __align__(16) unsigned char raw[];
    OneSmem& m = *reinterpret_cast<OneSmem*>(raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t a0 = (int32_t)min((int64_t)blockIdx.x * per_block, n_nodes);
    const int own = (int)min((int64_t)per_block, n_nodes - a0);
    for (int i = threadIdx.x; i <= own; i += kOneThreads) m.start[i] = 0;
    if (threadIdx.x == 0) m.collected = m.before = 0;
    __syncthreads();
    fast::grid_dependency_wait();
    fast::grid_dependency_trigger();
    int32_t smaller = 0;
    for_senders(n_nodes, n_edges, senders, pad_recv, [&](int64_t e, int32_t s) {
        smaller += s < a0;
        if (s >= a0 && s < a0 + own) {
            const int32_t place = atomicAdd(&m.start[s - a0], 1), at = atomicAdd(&m.collected, 1);
            if (at < kOneCap) { m.edge[at] = (int32_t)e; m.node[at] = (s - a0) << 13 | place; }
        }
    });
    smaller = __reduce_add_sync(0xffffffffu, smaller);
    if (lane == 0 && smaller) atomicAdd(&m.before, smaller);
    if (rowptr)
        fill_rowptr(n_nodes, n_edges, receivers, rowptr, blockIdx.x * (int64_t)kOneThreads + threadIdx.x,
                    (int64_t)gridDim.x * kOneThreads);
    __syncthreads();
    // exclusive scan of the counters: a run of them per thread, then over the threads
    const int run = (own + kOneThreads - 1) / kOneThreads;
    const int i0 = min((int)threadIdx.x * run, own), i1 = min(i0 + run, own);
    int32_t mine = 0;
    for (int i = i0; i < i1; ++i) mine += m.start[i];
    int32_t incl = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int32_t up = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += up;
    }
    if (lane == 31) m.warp_sum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int32_t ws = m.warp_sum[lane];
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int32_t up = __shfl_up_sync(0xffffffffu, ws, off);
            if (lane >= off) ws += up;
        }
        m.warp_sum[lane] = ws;
    }
    __syncthreads();
    const int32_t base = m.before, n_own = m.collected;
    int32_t first = (warp ? m.warp_sum[warp - 1] : 0) + incl - mine;
    for (int i = i0; i < i1; ++i) {
        const int32_t c = m.start[i];
        m.start[i] = first;
        colptr[a0 + i] = base + first;
        first += c;
    }
    if (threadIdx.x == 0) {
        m.start[own] = n_own;
        if (a0 + own == n_nodes && own > 0) colptr[n_nodes] = base + n_own;
    }
    __syncthreads();
    if (n_own <= kOneCap) {
        for (int t = threadIdx.x; t < n_own; t += kOneThreads) {
            const int l = m.node[t] >> 13, to = m.start[l] + (m.node[t] & 8191);
            m.key[to] = m.edge[t];
            m.of[to] = l;
        }
        __syncthreads();
        // edge ids are distinct: an edge's place in its bucket is the number of smaller ones there
        for (int t = threadIdx.x; t < n_own; t += kOneThreads) {
            const int32_t key = m.key[t], b = m.start[m.of[t]], end = m.start[m.of[t] + 1];
            int32_t at = base + b;
            for (int j = b; j < end; ++j) at += m.key[j] < key;
            perm[at] = key;
        }
        return;
    }
    // more edges than fit (senders of very many edges): the buckets are filled in place from a second reading, with the
    // place kept in a counter of its own, and sorted there
    for (int i = threadIdx.x; i < own; i += kOneThreads) m.of[i] = 0;
    __syncthreads();
    for_senders(n_nodes, n_edges, senders, pad_recv, [&](int64_t e, int32_t s) {
        if (s >= a0 && s < a0 + own) perm[base + m.start[s - a0] + atomicAdd(&m.of[s - a0], 1)] = (int32_t)e;
    });
    __syncthreads();
    static_assert(4 * kOneCap == kOneWarps * kRankMax, "the collected edges' four arrays serve as staging");
    for (int i = warp; i < own; i += kOneWarps)
        sort_bucket<kRankMax>(perm + base + m.start[i], m.start[i + 1] - m.start[i],
                              reinterpret_cast<int32_t*>(raw) + kRankMax * warp);
}

int prepare_one(int64_t n_nodes, int64_t n_edges, const int32_t* senders, const int32_t* receivers,
                const int32_t* pad_recv, int32_t* rowptr, int32_t* sender_perm, int32_t* colptr, cudaStream_t st) {
    // 16 nodes a block (a thread or so per edge in the sort), fewer where 16 would have more than about 4096 edges, up
    // to 128 blocks, then equal runs
    const int64_t want = std::max((n_nodes + 15) / 16, std::min(n_nodes, (n_edges + 4095) / 4096));
    const int64_t blocks = std::min<int64_t>(kOneBlocks, want);
    const int per_block = (int)((n_nodes + blocks - 1) / blocks);
    static thread_local int attr_dev = -1;
    int dev = 0;
    E3J_CUDA_TRY(cudaGetDevice(&dev));
    if (attr_dev != dev) {
        E3J_CUDA_TRY(cudaFuncSetAttribute(prepare_one_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(OneSmem)));
        attr_dev = dev;
    }
    return launch_dependent(prepare_one_kernel, dim3((int)blocks), dim3(kOneThreads), sizeof(OneSmem), st, n_nodes, n_edges, senders,
                            receivers, pad_recv, rowptr, colptr, sender_perm, per_block);
}

inline int blocks_for(int64_t n, int threads) {
    int64_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > sm_count() * 16) b = sm_count() * 16;
    return (int)b;
}

}  // namespace

int graph_prepare(int64_t n_nodes, int64_t n_edges, const int32_t* senders, const int32_t* receivers,
                  int32_t* rowptr, int32_t* sender_perm, int32_t* colptr, cudaStream_t st, bool padded) {
    const int32_t* pad_recv = padded ? receivers : nullptr;
    if (sender_perm && colptr && n_edges > 0 && n_edges <= kOneLaunchEdges && n_nodes > 0 &&
        n_nodes <= (int64_t)kOneBlocks * kOneNodes)
        return prepare_one(n_nodes, n_edges, senders, receivers, pad_recv, rowptr, sender_perm, colptr, st);
    if (rowptr) {
        const int64_t items = n_nodes > kFillNodes ? n_nodes + 1 : std::max(n_nodes + 1, n_edges);
        rowptr_kernel<<<blocks_for(items, 256), 256, 0, st>>>(n_nodes, n_edges, receivers, rowptr);
        if (int s = after_launch()) return s;
    }
    if (sender_perm && colptr) {
        E3J_CUDA_TRY(cudaMemsetAsync(colptr, 0, sizeof(int32_t) * (size_t)(n_nodes + 1), st));
        if (n_edges > 0) {
            count_senders_kernel<<<blocks_for(n_edges, 256), 256, 0, st>>>(n_nodes, n_edges, senders, pad_recv, colptr);
            if (int s = after_launch()) return s;
        }
        exclusive_scan_kernel<<<1, 1024, 0, st>>>(n_nodes, colptr);
        if (int s = after_launch()) return s;
        if (n_edges > 0) {
            fill_kernel<<<blocks_for(n_edges, 256), 256, 0, st>>>(n_nodes, n_edges, senders, pad_recv, colptr,
                                                               sender_perm);
            if (int s = after_launch()) return s;
            sort_buckets_kernel<<<blocks_for(n_nodes, kSortWarps), 32 * kSortWarps, 0, st>>>(n_nodes, colptr, sender_perm);
            if (int s = after_launch()) return s;
            shift_up_kernel<<<1, 1024, 0, st>>>(n_nodes, colptr);
            if (int s = after_launch()) return s;
        }
    }
    return E3J_OK;
}

int graph_validate(int64_t n_nodes, int64_t n_edges, const int32_t* senders, const int32_t* receivers,
                   int32_t* status, cudaStream_t st) {
    E3J_CUDA_TRY(cudaMemsetAsync(status, 0, sizeof(int32_t), st));
    if (n_edges > 0) {
        validate_kernel<<<blocks_for(n_edges, 256), 256, 0, st>>>(n_nodes, n_edges, senders, receivers, status);
        if (int s = after_launch()) return s;
    }
    return E3J_OK;
}

}  // namespace e3j
