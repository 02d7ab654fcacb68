#include "path_launch.cuh"

namespace e3j {
namespace path {

bool covers(const e3j_plan* plan, int vec) {
    if (plan->nq % vec != 0 || plan->nq / vec > kThreads) return false;
    for (const e3j_path_info_t& p : plan->paths)
        if (p.l1 > 3 || p.l2 > 3 || p.L > 3) return false;
    int extra = 0;
    for_unread_rows(plan, [&](int, int) { ++extra; });
    return plan->dp <= 16 && plan->P + extra <= 255;
}

int conv_fwd(const e3j_plan* plan, const Call<float>& c, bool ident) {
    if (ident) { E3J_BY_LARGEST_L(fwd, float, 4, true) }
    E3J_BY_LARGEST_L(fwd, float, 4, false)
}
int conv_bwd(const e3j_plan* plan, const Call<float>& c, bool ident) {
    if (ident) { E3J_BY_LARGEST_L(bwd, float, 4, true) }
    E3J_BY_LARGEST_L(bwd, float, 4, false)
}

}  // namespace path
}  // namespace e3j
