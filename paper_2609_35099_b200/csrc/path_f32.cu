#include "path_launch.cuh"

namespace e3j {
namespace path {

bool covers(const e3j_plan* plan, int vec) {
    return plan->path.covered && plan->nq % vec == 0 && plan->nq / vec <= kThreads;
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
