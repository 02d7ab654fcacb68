#include "path_table.hpp"

#include <algorithm>
#include <vector>

#include "plan.hpp"

namespace e3j {
namespace path {
namespace {

// Input rows that no path reads (an irrep whose products the output filter drops), cut into groups of 7, 5, 3 or 1
// rows: f(first row, l of a block of that size).  Their grad_x is zero.
template <class F> void for_unread_rows(const e3j_plan& plan, F f) {
    constexpr int kMaxDeg = 7;
    std::vector<char> read(plan.d, 0);
    for (const e3j_path_info_t& p : plan.paths) std::fill_n(read.begin() + p.x_off, 2 * p.l1 + 1, 1);
    for (int row = 0; row < plan.d;) {
        int n = 0;
        while (n < kMaxDeg && row + n < plan.d && !read[row + n]) ++n;
        if (n) f(row, (n - 1) / 2);
        row += n ? 2 * ((n - 1) / 2) + 1 : 1;
    }
}

enum class Group { kOutput, kInput, kPair };

// Paths grouped by output block (forward), by input block (backward), or by input block and harmonic degree (forward);
// a group's paths in plan order, those of a pair by L.
void fill_table(const e3j_plan& plan, Group by, int largest_l, PathTable& t) {
    t.n_paths = plan.P;
    std::vector<int> order(plan.P);
    for (int k = 0; k < plan.P; ++k) order[k] = k;
    auto key = [&](int k) {
        const e3j_path_info_t& pi = plan.paths[k];
        if (by == Group::kOutput) return pi.out_off;
        if (by == Group::kInput) return pi.x_off;
        return pi.x_off * 64 + pi.l2 * 8 + (largest_l == 3 && pi.L == 3 ? 4 : 0);   // paths to L = 3: groups of their own (registers)
    };
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        return by == Group::kPair && key(a) == key(b) ? plan.paths[a].L < plan.paths[b].L : key(a) < key(b);
    });
    for (int p = 0; p < plan.P; ++p) {
        const int k = order[p];
        const e3j_path_info_t& pi = plan.paths[k];
        t.rec[p] = PathRec{(uint8_t)tri_id(pi.l1, pi.l2, pi.L), (uint8_t)pi.l1, (uint8_t)pi.L, (uint8_t)k,
                           (uint8_t)pi.x_off, (uint8_t)pi.y_off, (uint8_t)pi.out_off, 0};
        if (p == 0 || key(k) != key(order[p - 1])) t.start[t.n_groups++] = (uint8_t)p;
    }
    int n = plan.P;
    if (by == Group::kInput)
        for_unread_rows(plan, [&](int row, int l) {
            t.rec[n] = PathRec{kNoPath, (uint8_t)l, 0, 0, (uint8_t)row, 0, 0, 0};
            t.start[t.n_groups++] = (uint8_t)n++;
        });
    t.start[t.n_groups] = (uint8_t)n;
}

void fill_edge_table(const PathTable& t, size_t row_bytes, EdgeTable& e) {
    e.n_paths = t.n_paths;
    for (int g = 0; g < t.n_groups; ++g)
        for (int p = t.start[g]; p < t.start[g + 1]; ++p) {
            const PathRec& r = t.rec[p];
            e.rec[e.n_recs++] = EdgeRec{(uint32_t)(r.k * row_bytes), (uint32_t)(r.out_off * row_bytes), (uint32_t)(r.x_off * row_bytes),
                                        r.id, (uint8_t)(2 * r.L + 1), (uint8_t)(p == t.start[g] ? 2 * r.l1 + 1 : 0), 0};
        }
}

}  // namespace

void build_path_plan(const e3j_plan& plan, PathPlan& out) {
    out = PathPlan{};
    int l = 1;
    while ((l + 1) * (l + 1) < plan.dp) ++l;
    for (const e3j_path_info_t& p : plan.paths) l = std::max({l, p.l1, p.l2, p.L});
    int extra = 0;
    for_unread_rows(plan, [&](int, int) { ++extra; });
    if (l > 3 || plan.P + extra > 255) return;
    fill_table(plan, Group::kOutput, l, out.by_output);
    fill_table(plan, Group::kInput, l, out.by_input);
    fill_table(plan, Group::kPair, l, out.by_pair);
    fill_edge_table(out.by_input, sizeof(float) * plan.nq, out.edges_f32);
    fill_edge_table(out.by_input, sizeof(double) * plan.nq, out.edges_f64);
    out.shared_rows = out.by_output.n_groups < plan.P;
    out.largest_l = l;
    for (const e3j_path_info_t& p : plan.paths) out.largest_l1 = std::max(out.largest_l1, p.l1);
    out.covered = true;
}

}  // namespace path
}  // namespace e3j
