// Force kernels of the FP64 form.
#include "force_launch.cuh"

namespace ljmd {

// Force over the list in the FP64 form, tile by tile (single buffer: the copies of a tile overlap the
// arithmetic of the SM's other three CTAs).  Bound by the FP64 pipe (77 % busy): 23 operations per pair
// inside r_c with energies, where every listed pair (1.7 times as many) took 29 in partly idle
// warps before.  The energies come from three sums over pairs (r^-6, r^-12, r^2) and their number.
// 1,048,576 particles, rho 0.5, half list, energies: 2.75 -> 1.03 ms per launch (T = 4 cells per tile;
// 3, 5 and 6 give 1.07, 1.14 and 1.05 ms); 4,000 particles 42 -> 24 us.
template <bool HALF, bool ENERGY>
__global__ void __launch_bounds__(kDpThreads, 4)
    k_force_dp(const dvec4* __restrict__ pos, const uint32_t* __restrict__ cs, Geom g, TileArgs ta, LJConst c,
               const uint2* __restrict__ rows, const uint2* __restrict__ tile_list, const uint16_t* __restrict__ ent,
               dvec4* __restrict__ fout, double* __restrict__ part, int32_t* __restrict__ status,
               const int* __restrict__ skip) {
  if (skip && *skip) return;  // a device-decided run stopped before this step
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ TileShared S;
  __shared__ __align__(8) uint64_t bar;
  const DpLayout D = dp_layout<3, HALF>(ta);
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_proxy_async_smem();
  }
  __syncthreads();
  DpForce<HALF, ENERGY> body(c, smem, D, fout);
  double npairs = 0.0;
  uint32_t ph = 0;
  for (int64_t t = blockIdx.x; t < ta.ntiles; t += gridDim.x) {
    const TileInfo ti = tile_info(t, ta);
    if (force_tile_prepare(ti, t, ta, cs, tile_list, S, status)) {
      stage_issue<false, true>(ti, ta, pos, rows, ent, S, smem, D.L, &bar);
      if (!dp_stage_finish(ti, ta, g, S, smem, D, &bar, ph, status)) return;
      auto pair = [&](const dvec4& qi, int j, double* acc) { body.pair(qi, j, acc); };
      auto done = [&](int o, const double* acc) {
        if (HALF) body.add(S.gown0 + o, acc);
        else fout[S.gown0 + o] = make_dvec4(acc[0], acc[1], acc[2], 0.0);
      };
      dp_tile_pairs<3, HALF>(S, smem, D, ent + S.list_base, (unsigned)ta.list_cap, body.cut2, status, pair, done);
      if (ENERGY) {
        npairs += (double)body.np;
        body.np = 0;
      }
    }
    __syncthreads();
  }
  if (ENERGY) {
    __shared__ double sh[32];
    double pe, vir;
    dp_energies(c, body.s6, body.s12, body.s2, npairs, pe, vir);
    const double tp = block_sum(pe, sh);
    __syncthreads();
    const double tv = block_sum(vir, sh);
    if (threadIdx.x == 0) {
      part[2 * (size_t)blockIdx.x] = tp;
      part[2 * (size_t)blockIdx.x + 1] = tv;
    }
  }
}

size_t dp_force_smem_bytes(const TileArgs& ta, int half) {
  return half ? dp_layout<3, true>(ta).total : dp_layout<3, false>(ta).total;
}
// Whether a CTA can stage the largest tile with its fixed-point records and queues (48 B per staged
// particle and 11 KB; about 4,600 particles).  Larger tiles (36 B per particle) take k_force_tile.
bool dp_fits(const TileArgs& ta) {
  int dev = 0, smem_max = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  TileArgs tz = ta;
  tz.list_cap = 0;
  return dp_layout<3, false>(tz).total + kStaticSmem <= (size_t)smem_max;
}

// The FP64 form on tiles; returns the grid launched.
template <bool HALF, bool ENERGY>
static int launch_dp(const ForceLaunch& a, size_t sm) {
  set_smem(k_force_dp<HALF, ENERGY>, sm);
  const int grid =
      tile_grid(a.ta, a.per_sm > 0 ? a.per_sm : resident_per_sm(k_force_dp<HALF, ENERGY>, kDpThreads, sm));
  k_force_dp<HALF, ENERGY><<<grid, kDpThreads, sm, a.s>>>((const dvec4*)a.pos, a.cs, a.g, a.ta, a.c, a.rows,
                                                           a.tile_list, a.ent, (dvec4*)a.f, a.part, a.status, a.skip);
  return grid;
}
static int launch_force_dp(int half, const ForceLaunch& a) {
  const size_t sm = dp_force_smem_bytes(a.ta, half);
  if (half) return a.energy ? launch_dp<true, true>(a, sm) : launch_dp<true, false>(a, sm);
  return a.energy ? launch_dp<false, true>(a, sm) : launch_dp<false, false>(a, sm);
}

template <bool HALF>
static void force_fp64_general(const ForceLaunch& a) {
  if (a.ta.whole) force_tile_lanes<false, HALF, true, false>(a);
  else force_tile_energy<false, HALF, false, true, 8>(a);  // tiles beyond k_force_dp's capacity
}

int launch_force_fp64(int half, ForceLaunch& a) {
  if (!a.ta.whole && dp_fits(a.ta)) return launch_force_dp(half, a);
  if (half) force_fp64_general<true>(a);
  else force_fp64_general<false>(a);
  return a.grid;
}
int set_wait_budget_force_dp(long long cycles) { return set_unit_wait_budget(cycles); }

}  // namespace ljmd
