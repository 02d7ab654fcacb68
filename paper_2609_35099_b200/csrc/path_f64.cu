#include "path_launch.cuh"

namespace e3j {
namespace path {

int conv_fwd(const e3j_plan* plan, const Call<double>& c) { E3J_BY_LARGEST_L(fwd, double, 2, false) }
int conv_bwd(const e3j_plan* plan, const Call<double>& c) { E3J_BY_LARGEST_L(bwd, double, 2, false) }

}  // namespace path
}  // namespace e3j
