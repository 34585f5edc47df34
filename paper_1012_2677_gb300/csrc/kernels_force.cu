// Force kernels of the mixed form with the full list (pipelined and single buffer), the batched
// replicas' force, and the dispatch over the forms.
#include "force_launch.cuh"

namespace ljmd {

// Shared memory of the force kernel: `nbuf` tile buffers (two: the least that the pipelined kernel takes); one
// for the whole-box case.
size_t force_buffer_bytes(const TileArgs& ta, int precision, int half) {
  const bool mixed = precision == LJ_MIXED;
  return align16(tile_layout(ta, mixed, true, !mixed && (half || ta.whole)).total);
}
size_t force_smem_bytes(const TileArgs& ta, int precision, int nbuf, int half) {
  if (precision != LJ_MIXED && !ta.whole) return dp_fits(ta) ? dp_force_smem_bytes(ta, half) : force_buffer_bytes(ta, precision, half);
  return (ta.whole ? 1 : (nbuf == 2 ? 2 : 1)) * force_buffer_bytes(ta, precision, half);
}

// ---------------------------------------------------------------------------------------------
// Batched replicas (mixed form, full list): one persistent launch walks the tiles of all
// replicas; each tile takes its replica's box and grid from the replica table.  Energies: the
// tile's PE and virial are reduced over the CTA and added to its replica's totals (e_rep[2 r],
// e_rep[2 r + 1]).
template <int LANES, bool ENERGY>
__global__ void __launch_bounds__(kTileThreads, 4)
    k_force_batch(const uint4* __restrict__ pos, const uint32_t* __restrict__ cs_in, int64_t N, TileArgs caps,
                  LJConst c, const uint2* __restrict__ rows,
                  const uint2* __restrict__ tile_list, const uint16_t* __restrict__ ent, float4* __restrict__ fout,
                  double* __restrict__ e_rep, int32_t* __restrict__ status, const ReplicaGeo* __restrict__ reps,
                  int R, const int32_t* __restrict__ tile_rep) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ TileShared S;
  __shared__ __align__(8) uint64_t bar;
  __shared__ double sh[32];
  const TileLayout L = tile_layout(caps, true, true, false);
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_proxy_async_smem();
  }
  __syncthreads();
  uint32_t ph = 0;
  for (int64_t t = blockIdx.x; t < caps.ntiles; t += gridDim.x) {
    const int r = tile_rep[t];
    const ReplicaGeo& rg = reps[r];
    TileArgs ta = caps;
    Geom g;
    replica_view(rg, ta, g);
    const uint32_t* cs = cs_in + rg.cell_base;
    const TileInfo ti = tile_info(t - rg.tile_base, ta);
    EAcc eacc;
    eacc.vscale = g.qu;
    if (force_tile_prepare(ti, t, ta, cs, tile_list, S, status)) {
      stage_issue<true, true>(ti, ta, pos, rows, ent, S, smem, L, &bar);
      if (!stage_finish<true, true>(ti, ta, g, S, smem, L, &bar, ph, false, status)) return;
      force_tile_compute<true, LANES, false, ENERGY, false, true>(S, smem, L, rows, ent, c, g, fout, status, eacc,
                                                                  ta.list_cap);
    }
    if (ENERGY) {
      eacc.flush();
      const double tp = block_sum(eacc.pe, sh);
      __syncthreads();
      const double tv = block_sum(eacc.vir, sh);
      if (threadIdx.x == 0) {
        atomicAdd(&e_rep[2 * r], 0.5 * tp);  // full list: each pair twice
        atomicAdd(&e_rep[2 * r + 1], 0.5 * tv);
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------------
// Buffers of the pipelined kernel for these tiles (0: not even two fit) and the entries of a segment
// that each stages: four, as long as they hold three quarters of the longest segment, else fewer.
int pipe_plan(TileArgs& ta) {
  int dev = 0, smem_max = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  TileArgs tz = ta;
  tz.list_cap = 0;
  const int64_t fixed = (int64_t)align16(tile_layout(tz, true, true, false).total);
  for (int nb = 4; nb >= 2; --nb) {
    const int64_t per = ((int64_t)smem_max - 1024) / nb & ~(int64_t)15;
    if (per < fixed) continue;
    const int64_t cap = std::min<int64_t>((per - fixed) / 2, ta.max_list) & ~(int64_t)7;
    if (nb > 2 && 4 * cap < 3 * (int64_t)ta.max_list) continue;
    ta.list_cap = (int32_t)cap;
    return nb;
  }
  return 0;
}

int launch_force_tile(int precision, int half, int lanes, int energy, const void* pos, const uint32_t* cs, int64_t N,
                      Geom g, TileArgs ta, LJConst c, const uint2* rows, const uint2* tile_list, const uint16_t* ent,
                      void* f, double* part, int32_t* status, int per_sm, int nbuf, cudaStream_t s, const int* skip,
                      bool overlap) {
  ForceLaunch a{pos, cs, N, g, ta, c, rows, tile_list, ent, f, part, status, skip, lanes, energy, per_sm, 1, 0, 0, s};
  a.overlap = overlap ? 1 : 0;
  a.smem = force_smem_bytes(ta, precision, 1, half);
  a.grid = tile_grid(ta, per_sm > 0 ? per_sm : per_sm_for(a.smem));
  if (precision != LJ_MIXED) return launch_force_fp64(half, a);
  if (!ta.whole && nbuf == 2 && (a.nbuf = pipe_plan(a.ta)) > 0) {
    if (half) {
      const int grid = launch_force_pipe_half(a);
      if (grid > 0) return grid;
    } else {
      switch (lanes) {
        case 1: return force_pipe_energy<false, 1>(a);
        case 2: return force_pipe_energy<false, 2>(a);
        case 4: return force_pipe_energy<false, 4>(a);
        case 8: return force_pipe_energy<false, 8>(a);
        case 16: return force_pipe_energy<false, 16>(a);
        default: return force_pipe_energy<false, 32>(a);
      }
    }
  }
  a.ta = ta;
  if (half) launch_force_mixed_half(a);
  else force_tile_mixed<false>(a);
  return a.grid;
}

size_t batch_force_smem_bytes(const TileArgs& caps) { return align16(tile_layout(caps, true, true, false).total); }

int launch_force_batch(int lanes, int energy, const uint4* xq, const uint32_t* cs, int64_t N,
                       TileArgs caps, LJConst c, const uint2* rows, const uint2* tile_list, const uint16_t* ent,
                       float4* f, double* e_rep, int32_t* status, const ReplicaGeo* reps, int R,
                       const int32_t* tile_rep, cudaStream_t s) {
  if (!energy) {  // the steps: the pipelined kernel over the tiles of all replicas
    ForceLaunch a{xq, cs, N, Geom{}, caps, c, rows, tile_list, ent, f, nullptr, status, nullptr, lanes, 0, 0, 0, 0, 0, s};
    a.nbuf = pipe_plan(a.ta);
    if (a.nbuf > 0) {
      switch (lanes) {
        case 2: return force_pipe<false, 2, false>(a);
        case 8: return force_pipe<false, 8, false>(a);
        default: return force_pipe<false, 4, false>(a);
      }
    }
  }
  const size_t sm = batch_force_smem_bytes(caps);
  const int grid = tile_grid(caps, per_sm_for(sm));
#define LJ_FB(LN)                                                                                               \
  do {                                                                                                          \
    if (energy) {                                                                                               \
      set_smem(k_force_batch<LN, true>, sm);                                                                    \
      k_force_batch<LN, true><<<grid, kTileThreads, sm, s>>>(xq, cs, N, caps, c, rows, tile_list, ent, f,       \
                                                             e_rep, status, reps, R, tile_rep);                          \
    } else {                                                                                                    \
      set_smem(k_force_batch<LN, false>, sm);                                                                   \
      k_force_batch<LN, false><<<grid, kTileThreads, sm, s>>>(xq, cs, N, caps, c, rows, tile_list, ent, f,      \
                                                              e_rep, status, reps, R, tile_rep);                         \
    }                                                                                                           \
  } while (0)
  switch (lanes) {
    case 2: LJ_FB(2); break;
    case 8: LJ_FB(8); break;
    default: LJ_FB(4); break;
  }
#undef LJ_FB
  return grid;
}

int set_wait_budget_force(long long cycles) { return set_unit_wait_budget(cycles); }

}  // namespace ljmd
