// The pipelined force kernel that also takes the step after the force (mixed form, full list).  The integrator
// by itself is bound by HBM (2.4 GB at 16.4M particles: 498 us) or, where the state is in L2, by its launch and
// its loads' latency (28 us at 500,000), and the force kernel by issue: together a step takes 1.69 ms instead of
// 1.82 at 16.4M particles, rho 0.5, with energies, and 73 us instead of 83 at 500,000 without.
// What was slower: the step by the threads of a key as its force is done (two thirds of the lanes, twice the
// instructions: 76 us at 500,000), by the producer warps (one warp's chain of 470 instructions per 32
// particles is longer than a tile lasts: 98 us).
#include "force_launch.cuh"

namespace ljmd {

bool step_pipe_lanes(int lanes) { return lanes == 2 || lanes == 4; }
int launch_step_pipe(const ForceLaunch& a) {
  return a.lanes == 2 ? force_pipe_energy<false, 2, true>(a) : force_pipe_energy<false, 4, true>(a);
}
int set_wait_budget_step(long long cycles) { return set_unit_wait_budget(cycles); }

}  // namespace ljmd
