// Internal: the path lists of the per-path kernels (path_kernels.cuh), formed with the plan.
#pragma once
#include <cstdint>

struct e3j_plan;

namespace e3j {
namespace path {

constexpr int tri_id(int l1, int l2, int L) { return l1 * 16 + l2 * 4 + L; }
constexpr uint8_t kNoPath = 255;   // a group of input rows that no path reads: nothing to add

// One plan's paths in a processing order, passed by value (kernel parameters: constant-bank reads, nothing to upload).
struct PathRec { uint8_t id, l1, L, k, x_off, y_off, out_off, pad; };
struct PathTable {
    int n_paths = 0, n_groups = 0;
    uint8_t start[257] = {};     // groups of paths that share the rows they are summed into
    PathRec rec[255] = {};
};
static_assert(sizeof(PathTable) < 3072, "the table travels in the kernel parameters");

// The backward's list as the edge part reads it: byte offsets into an edge's rows.  A path costs the edge part about a
// hundred integer instructions less than with the offsets formed there (48x(0e+1o+2e), l <= 2, 35 050 edges, with the
// sum of the shares: 133 -> 106 us).
struct EdgeRec {
    uint32_t w, g, x;             // the path's weights, its first grad_out row, the first row of its input block
    uint8_t id, n_g, n_x, pad;    // rows of grad_out; rows of the input block if it is the first path there, else 0
};
struct EdgeTable {
    int n_paths = 0, n_recs = 0;  // records behind n_paths: input rows that no path reads, n_x of them from x
    EdgeRec rec[255] = {};
};

// What the per-path kernels need to know of a plan.  Formed once, at plan creation: a call neither allocates host
// memory (whose failure would leave the C interface as an exception) nor repeats the work.
struct PathPlan {
    bool covered = false;        // every l <= 3, and the groups fit a table
    int largest_l = 0, largest_l1 = 0;
    bool shared_rows = false;    // some output block has several paths
    PathTable by_output, by_input, by_pair;
    EdgeTable edges_f32, edges_f64;
};
void build_path_plan(const e3j_plan& plan, PathPlan& out);

}  // namespace path
}  // namespace e3j
