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

// Paths in plan order, grouped by output block (forward), or by input block (backward).
void fill_table(const e3j_plan& plan, bool by_input, PathTable& t) {
    t.n_paths = plan.P;
    std::vector<int> order(plan.P);
    for (int k = 0; k < plan.P; ++k) order[k] = k;
    auto key = [&](int k) { return by_input ? plan.paths[k].x_off : plan.paths[k].out_off; };
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return key(a) < key(b); });
    for (int p = 0; p < plan.P; ++p) {
        const int k = order[p];
        const e3j_path_info_t& pi = plan.paths[k];
        t.rec[p] = PathRec{(uint8_t)tri_id(pi.l1, pi.l2, pi.L), (uint8_t)pi.l1, (uint8_t)pi.L, (uint8_t)k,
                           (uint8_t)pi.x_off, (uint8_t)pi.y_off, (uint8_t)pi.out_off, 0};
        if (p == 0 || key(k) != key(order[p - 1])) t.start[t.n_groups++] = (uint8_t)p;
    }
    int n = plan.P;
    if (by_input)
        for_unread_rows(plan, [&](int row, int l) {
            t.rec[n] = PathRec{kNoPath, (uint8_t)l, 0, 0, (uint8_t)row, 0, 0, 0};
            t.start[t.n_groups++] = (uint8_t)n++;
        });
    t.start[t.n_groups] = (uint8_t)n;
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
    fill_table(plan, false, out.by_output);
    fill_table(plan, true, out.by_input);
    out.largest_l = l;
    out.covered = true;
}

}  // namespace path
}  // namespace e3j
