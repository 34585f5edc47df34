// Force kernels of the mixed form with the full list (pipelined and single buffer), the batched
// replicas' force, and the dispatch over the forms.
#include "force_launch.cuh"

namespace ljmd {

// Shared memory of the force kernel: `nbuf` tile buffers (with two, the next tile's copies are in
// flight while the current one is computed); one for the whole-box case.
size_t force_buffer_bytes(const TileArgs& ta, int precision, int half) {
  const bool mixed = precision == LJ_MIXED;
  return align16(tile_layout(ta, mixed, true, !mixed && (half || ta.whole)).total);
}
size_t force_smem_bytes(const TileArgs& ta, int precision, int nbuf, int half) {
  if (precision != LJ_MIXED && !ta.whole) return dp_fits(ta) ? dp_force_smem_bytes(ta, half) : force_buffer_bytes(ta, precision, half);
  return (ta.whole ? 1 : (nbuf == 2 ? 2 : 1)) * force_buffer_bytes(ta, precision, half);
}

// ---------------------------------------------------------------------------------------------
// Pipelined force (mixed form, full list, tiled box): two producer warps stage tiles into two
// shared-memory buffers (producer p handles the tiles k = p mod 2, in buffer p) while the consumer
// warps compute, so neither the copies nor the tile-end stragglers hold the CTA at a barrier.
// Per tile k (buffer k % 2, bookkeeping slot k % 4):
//   producer: wait empty[b] (tile k - 2 released) -> issue the copies of tile k -> bookkeeping of
//             tile k + 2 from cell bounds loaded one tile earlier, and the loads for tile k + 4 ->
//             wait full[b] -> arrive ready[b];
//   consumers: wait ready[b] -> (periodic tiles: image shifts, consumer barrier) -> forces of
//             the tile's own particles -> arrive empty[b].
// Every wait is bounded; a producer that gives up marks the slot aborted and releases the
// consumers, which then leave.  No copy is in flight when a warp leaves.
constexpr int kPipeProducers = 2;
constexpr int kPipeSlots = 4;
__host__ __device__ constexpr int pipe_threads(int cw) { return 32 * (cw + kPipeProducers); }

__device__ __forceinline__ bool tile_interior(const TileInfo& ti, const TileArgs& ta) {
  return ti.cx >= 1 && ti.cx <= ta.n - 2 && ti.cy >= 1 && ti.cy <= ta.n - 2 && ti.z0 >= 1 && ti.z0 + ti.Tp <= ta.n - 1;
}

// Image shifts of a staged tile's periodic cells by the consumer warps (warp per cell, lanes over
// its particles): integer adds of round(L / u) to the fixed-point records.  Every writer orders its
// writes before later bulk copies into the same bytes; the caller then waits for all consumer
// warps (a bounded mbarrier wait, not bar.sync, so that a warp that left on a timeout cannot hold
// the others forever).
__device__ __forceinline__ void stage_shift_consumers(const TileInfo& ti, const TileArgs& ta, const Geom& g,
                                                      const TileShared& S, unsigned char* smem, const TileLayout& L,
                                                      int consumers) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int q = warp; q < S.ncell; q += consumers) {
    int sx, sy, sz;
    cell_of_q(ti, ta.n, S.ncol, q, sx, sy, sz);
    if ((sx | sy | sz) == 0) continue;
    for (int e = S.offq[q] + lane; e < S.offq[q + 1]; e += 32) {
      uint4* r = (uint4*)(smem + L.pos) + e;
      r->x = shift_q(r->x, sx, g);
      r->y = shift_q(r->y, sy, g);
      r->z = shift_q(r->z, sz, g);
    }
  }
  fence_proxy_async_smem();
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// CW consumer warps: 8 for tiles of up to 4 cells, 12 for larger tiles (more keys per tile).  The
// consumers put the periodic images of a boundary tile in place before computing it.
template <int LANES, bool ENERGY, bool LONGLIST, int CW>
__global__ void __launch_bounds__(pipe_threads(CW), CW <= 8 ? 3 : 2)
    k_force_pipe(const void* __restrict__ pos, const uint32_t* __restrict__ cs, Geom g, TileArgs ta, LJConst c,
                 const uint2* __restrict__ rows, const uint2* __restrict__ tile_list,
                 const uint16_t* __restrict__ ent, void* __restrict__ fout, double* __restrict__ part,
                 int32_t* __restrict__ status, const int* __restrict__ skip) {
  if (skip && *skip) return;  // a device-decided run stopped before this step
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ TileShared SS[kPipeSlots];
  __shared__ TileInfo s_ti[kPipeSlots];
  __shared__ int s_valid[kPipeSlots];  // 1: interior tile, 2: periodic tile (shifts), 0: skip, -1: abort
  __shared__ __align__(8) uint64_t full[2], ready[2], empty[2], shifted[2];
  const TileLayout L = tile_layout(ta, true, true, false);
  const size_t buf_bytes = align16(L.total);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(&full[b], 1);
      mbar_init(&ready[b], 1);
      mbar_init(&empty[b], CW);
      mbar_init(&shifted[b], CW);
    }
    fence_proxy_async_smem();
  }
  __syncthreads();
  EAcc eacc;
  eacc.vscale = g.qu;
  const int64_t stride = gridDim.x;
  if (warp >= CW) {
    // ---- producer p: tiles k = p, p + 2, ... in buffer p ----
    const int p = warp - CW, b = p;
    int64_t t = blockIdx.x + p * stride;
    TilePrefetch pf;
    bool ok_next = false;
    TileInfo ti_cur{0, 0, 0, 0};
    if (t < ta.ntiles) {
      tile_prefetch(t, ta, cs, tile_list, pf, lane);
      ti_cur = pf.ti;
      ok_next = tile_prepare_pf(pf, ta, SS[p], lane);
      if (t + 2 * stride < ta.ntiles) tile_prefetch(t + 2 * stride, ta, cs, tile_list, pf, lane);
    }
    for (int k = p; t < ta.ntiles; t += 2 * stride, k += 2) {
      const int slot = k % kPipeSlots;
      const uint32_t use = (uint32_t)(k >> 1);
      TileShared& S = SS[slot];
      unsigned char* buf = smem + b * buf_bytes;
      bool ok = true;
      if (k >= 2) {
        if (lane == 0) ok = mbar_wait(&empty[b], (use - 1u) & 1u, wait_budget());
        ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
      }
      if (!ok) {  // the consumers did not release the buffer: give up (nothing in flight)
        if (lane == 0) {
          atomicOr(status, LJ_ST_TIMEOUT);
          s_valid[slot] = -1;
          mbar_arrive(&ready[b]);
        }
        break;
      }
      const TileInfo ti = ti_cur;
      bool staged = ok_next;
      if (staged && (S.own1 - S.own0 > ta.max_own || S.list_len > (unsigned)ta.max_list)) {
        if (lane == 0) atomicOr(status, LJ_ST_LIST_OVERFLOW);
        staged = false;
      }
      if (!staged && lane == 0 && !ok_next) atomicOr(status, LJ_ST_CELL_RANGE);
      if (staged) stage_issue<true, true>(ti, ta, pos, rows, ent, S, buf, L, &full[b], warp);
      // bookkeeping of this producer's next tile (its slot was released with tile k - 2), then
      // the loads for the one after it
      const int64_t tn = t + 2 * stride;
      if (tn < ta.ntiles) {
        ti_cur = pf.ti;
        ok_next = tile_prepare_pf(pf, ta, SS[(k + 2) % kPipeSlots], lane);
        if (tn + 2 * stride < ta.ntiles) tile_prefetch(tn + 2 * stride, ta, cs, tile_list, pf, lane);
      }
      if (staged) {
        bool landed = true;
        if (lane == 0) landed = mbar_wait(&full[b], use & 1u, wait_budget());
        landed = __shfl_sync(0xffffffffu, landed ? 1 : 0, 0) != 0;
        if (!landed) {
          if (lane == 0) {
            atomicOr(status, LJ_ST_TIMEOUT);
            mbar_wait(&full[b], use & 1u, kWaitBudget);  // let copies in flight land before leaving
            s_valid[slot] = -1;
            mbar_arrive(&ready[b]);
          }
          break;
        }
      }
      if (lane == 0) {
        s_ti[slot] = ti;
        s_valid[slot] = staged ? (tile_interior(ti, ta) ? 1 : 2) : 0;
        mbar_arrive(&ready[b]);  // release: bookkeeping and copies visible to the consumers
      }
    }
  } else {
    // ---- consumers ----
    int k = 0;
    uint32_t shpar = 0u;  // bit b: phase of shifted[b] (every consumer warp sees the same tiles)
    for (int64_t t = blockIdx.x; t < ta.ntiles; t += stride, ++k) {
      const int b = k & 1, slot = k % kPipeSlots;
      const uint32_t use = (uint32_t)(k >> 1);
      bool ok = __all_sync(0xffffffffu, mbar_wait(&ready[b], use & 1u, wait_budget())) != 0;
      if (!ok) {
        if (lane == 0) atomicOr(status, LJ_ST_TIMEOUT);
        break;
      }
      const int v = s_valid[slot];
      if (v < 0) break;
      unsigned char* buf = smem + b * buf_bytes;
      if (v == 2) {  // periodic tile: shifts by all consumer warps, then wait for all of them
        stage_shift_consumers(s_ti[slot], ta, g, SS[slot], buf, L, CW);
        __syncwarp();
        if (lane == 0) mbar_arrive(&shifted[b]);
        ok = __all_sync(0xffffffffu, mbar_wait(&shifted[b], (shpar >> b) & 1u, wait_budget())) != 0;
        shpar ^= 1u << b;
        if (!ok) {
          if (lane == 0) atomicOr(status, LJ_ST_TIMEOUT);
          break;
        }
      }
      if (v > 0)
        force_tile_compute<true, LANES, false, ENERGY, false, LONGLIST, 32 * CW>(SS[slot], buf, L, rows, ent, c, g,
                                                                                    fout, status, eacc, ta.list_cap);
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[b]);
    }
  }
  __syncthreads();
  if (ENERGY) {
    __shared__ double sh[32];
    eacc.flush();
    const double tp = block_sum(eacc.pe, sh);
    __syncthreads();
    const double tv = block_sum(eacc.vir, sh);
    if (threadIdx.x == 0) {
      part[2 * (size_t)blockIdx.x] = tp;
      part[2 * (size_t)blockIdx.x + 1] = tv;
    }
  }
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
// The mixed form with the full list: the pipelined kernel (two buffers) or the single-buffer one.
// Both return the grid launched (the number of energy partials written).
template <int LANES, bool ENERGY, bool LONGLIST, int CW>
static int force_pipe_launch(const ForceLaunch& a) {
  set_smem(k_force_pipe<LANES, ENERGY, LONGLIST, CW>, a.smem);
  const int64_t want =
      (int64_t)sm_count() * resident_per_sm(k_force_pipe<LANES, ENERGY, LONGLIST, CW>, pipe_threads(CW), a.smem);
  const int grid =
      (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(want, a.ta.ntiles), (int64_t)kMaxRedBlocks));
  k_force_pipe<LANES, ENERGY, LONGLIST, CW><<<grid, pipe_threads(CW), a.smem, a.s>>>(
      a.pos, a.cs, a.g, a.ta, a.c, a.rows, a.tile_list, a.ent, a.f, a.part, a.status, a.skip);
  return grid;
}
template <int LANES, bool ENERGY>
static int force_pipe(const ForceLaunch& a) {
  const bool lg = a.ta.list_cap < a.ta.max_list;
  if (a.ta.T <= 4) return lg ? force_pipe_launch<LANES, ENERGY, true, 8>(a) : force_pipe_launch<LANES, ENERGY, false, 8>(a);
  return lg ? force_pipe_launch<LANES, ENERGY, true, 12>(a) : force_pipe_launch<LANES, ENERGY, false, 12>(a);
}
template <int LANES>
static int force_pipe_energy(const ForceLaunch& a) {
  return a.energy ? force_pipe<LANES, true>(a) : force_pipe<LANES, false>(a);
}

int launch_force_tile(int precision, int half, int lanes, int energy, const void* pos, const uint32_t* cs, int64_t N,
                      Geom g, TileArgs ta, LJConst c, const uint2* rows, const uint2* tile_list, const uint16_t* ent,
                      void* f, double* part, int32_t* status, int per_sm, int nbuf, cudaStream_t s, const int* skip) {
  ForceLaunch a{pos, cs, N, g, ta, c, rows, tile_list, ent, f, part, status, skip, lanes, energy, per_sm, nbuf, 0, 0, s};
  a.smem = force_smem_bytes(ta, precision, nbuf, half);
  a.grid = tile_grid(ta, per_sm > 0 ? per_sm : per_sm_for(a.smem));
  if (precision != LJ_MIXED) {
    if (!ta.whole) a.nbuf = 1;
    return launch_force_fp64(half, a);
  }
  if (half) {
    launch_force_mixed_half(a);
  } else if (!ta.whole && nbuf == 2) {
    switch (lanes) {
      case 1: return force_pipe_energy<1>(a);
      case 2: return force_pipe_energy<2>(a);
      case 4: return force_pipe_energy<4>(a);
      case 8: return force_pipe_energy<8>(a);
      case 16: return force_pipe_energy<16>(a);
      default: return force_pipe_energy<32>(a);
    }
  } else {
    force_tile_mixed<false>(a);
  }
  return a.grid;
}

size_t batch_force_smem_bytes(const TileArgs& caps) { return align16(tile_layout(caps, true, true, false).total); }

int launch_force_batch(int lanes, int energy, const uint4* xq, const uint32_t* cs, int64_t N,
                       TileArgs caps, LJConst c, const uint2* rows, const uint2* tile_list, const uint16_t* ent,
                       float4* f, double* e_rep, int32_t* status, const ReplicaGeo* reps, int R,
                       const int32_t* tile_rep, cudaStream_t s) {
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
