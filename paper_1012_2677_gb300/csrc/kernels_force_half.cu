// Force kernel of the mixed form with the half list (Newton-3 scatter).
#include "force_launch.cuh"

namespace ljmd {

void launch_force_mixed_half(const ForceLaunch& a) { force_tile_mixed<true>(a); }
int set_wait_budget_force_half(long long cycles) { return set_unit_wait_budget(cycles); }

}  // namespace ljmd
