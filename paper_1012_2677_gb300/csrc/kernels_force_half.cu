// Force kernel of the mixed form with the half list (Newton-3 scatter).
#include "force_launch.cuh"

namespace ljmd {

void launch_force_mixed_half(const ForceLaunch& a) { force_tile_mixed<true>(a); }
// Returns the grid launched (0: the pipelined kernel is not built for this number of threads per key).
int launch_force_pipe_half(const ForceLaunch& a) {
  switch (a.lanes) {
    case 2: return force_pipe_energy<true, 2>(a);
    case 4: return force_pipe_energy<true, 4>(a);
    case 8: return force_pipe_energy<true, 8>(a);
    default: return 0;
  }
}
int set_wait_budget_force_half(long long cycles) { return set_unit_wait_budget(cycles); }

}  // namespace ljmd
