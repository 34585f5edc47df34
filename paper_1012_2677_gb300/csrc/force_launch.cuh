// The pipelined force kernel and the launches of it and of k_force_tile for one precision and list form:
// included by the translation unit that builds the form (one each, so that they compile in parallel).
#pragma once

#include "tile.cuh"

namespace ljmd {

template <bool MIXED, bool HALF, bool WHOLE, bool LONGLIST, int LANES, bool ENERGY>
static void force_tile_launch(const ForceLaunch& a) {
  set_smem(k_force_tile<MIXED, LANES, HALF, ENERGY, WHOLE, LONGLIST>, a.smem);
  k_force_tile<MIXED, LANES, HALF, ENERGY, WHOLE, LONGLIST><<<a.grid, kTileThreads, a.smem, a.s>>>(
      a.pos, a.cs, a.N, a.g, a.ta, a.c, a.rows, a.tile_list, a.ent, a.f, a.part, a.status, a.skip);
}

template <bool MIXED, bool HALF, bool WHOLE, bool LONGLIST, int LANES>
static void force_tile_energy(const ForceLaunch& a) {
  if (a.energy) force_tile_launch<MIXED, HALF, WHOLE, LONGLIST, LANES, true>(a);
  else force_tile_launch<MIXED, HALF, WHOLE, LONGLIST, LANES, false>(a);
}

template <bool MIXED, bool HALF, bool WHOLE, bool LONGLIST>
static void force_tile_lanes(const ForceLaunch& a) {
  switch (a.lanes) {
    case 1: force_tile_energy<MIXED, HALF, WHOLE, LONGLIST, 1>(a); break;
    case 2: force_tile_energy<MIXED, HALF, WHOLE, LONGLIST, 2>(a); break;
    case 4: force_tile_energy<MIXED, HALF, WHOLE, LONGLIST, 4>(a); break;
    case 8: force_tile_energy<MIXED, HALF, WHOLE, LONGLIST, 8>(a); break;
    case 16: force_tile_energy<MIXED, HALF, WHOLE, LONGLIST, 16>(a); break;
    default: force_tile_energy<MIXED, HALF, WHOLE, LONGLIST, 32>(a); break;
  }
}

// The mixed form: whole box, tiles with long segments, tiles.
template <bool HALF>
static void force_tile_mixed(const ForceLaunch& a) {
  if (a.ta.whole) force_tile_lanes<true, HALF, true, false>(a);
  else if (a.ta.list_cap < a.ta.max_list) force_tile_lanes<true, HALF, false, true>(a);  // some beyond the staged capacity
  else force_tile_lanes<true, HALF, false, false>(a);
}

// ---------------------------------------------------------------------------------------------
// Pipelined force (mixed form, tiled box): one CTA per SM, NB producer warps that stage
// tiles into NB shared-memory buffers (producer p handles the tiles k = p mod NB, in buffer p) and 24
// consumer warps that share the keys of all staged tiles, so neither the copies nor the tile-end
// stragglers hold anybody at a barrier.  Per tile k (buffer b = k % NB):
//   producer: wait empty[b] (tile k - NB released) -> issue the copies of tile k from its descriptor
//             (loaded one tile earlier) -> wait full[b] -> (boundary tiles: image shifts) -> arrive ready[b];
//   consumers: wait ready[b] -> forces of the warp's share of the tile's own particles -> arrive
//             empty[b].
// A tile beyond the capacities (a batch's device-side construction can make one) is recorded in the status
// word and skipped: it goes through ready and empty as any other, but nothing is copied and full[b]
// completes no phase, so the producer counts the buffer's fills apart from its uses.
// Every wait is bounded; a producer that gives up marks the slot aborted and releases the
// consumers, which then leave.  No copy is in flight when a warp leaves.
//
// Bound by issue (67 % busy) and by the latency of a warp's pair chain, so what counts is that all warps
// always have keys and that the producers, whose dependent instructions each wait their turn among 28
// warps, have little to do.  With a producer working out a tile's cell bounds and prefix sums (40 to 60 %
// of its time), two CTAs of two buffers, a tile's keys spread from the first warp on and scalar pair
// arithmetic, a launch took 2.01 ms at 16.4M particles, rho 0.5 (12 cells per tile), and 78 us at
// 500,000; now 1.32 ms and 55 us.  Packed arithmetic alone gave 1.92 ms, staging the front of long segments
// 1.86 ms, four buffers in one CTA 1.83 ms, the descriptors 1.32 ms.  The half list (2M particles, rho 0.8,
// single buffer before): 472 -> 276 us, of which 46 us for leaving out the atomics of pairs outside r_c.
constexpr int kPipeConsumers = 24;
__host__ __device__ constexpr int pipe_threads(int nb) { return 32 * (kPipeConsumers + nb); }

// What the consumers need of a staged tile.
struct PipeTile {
  int own0, own1, gown0, row_off;
  unsigned list_base, list_len;
  int valid;  // 1: staged, 0: skip, -1: abort
};

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Image shifts of a staged boundary tile by its producer warp (lane l holds run l: slot, particles and
// shift): integer adds of round(L / u) to the fixed-point records.
__device__ __forceinline__ void pipe_shift(uint4* rec, uint32_t run, uint32_t ax, uint32_t ay, uint32_t az, int lane) {
  unsigned m = __ballot_sync(0xffffffffu, (run & 0xffffu) != 0u && (ax | ay | az) != 0u);
  while (m) {
    const int l = __ffs(m) - 1;
    m &= m - 1;
    const uint32_t w = __shfl_sync(0xffffffffu, run, l);
    const uint32_t bx = __shfl_sync(0xffffffffu, ax, l), by = __shfl_sync(0xffffffffu, ay, l),
                   bz = __shfl_sync(0xffffffffu, az, l);
    uint4* q = rec + (w >> 16);
    const int n = (int)(w & 0xffffu);
#pragma unroll 4
    for (int e = lane; e < n; e += 32) {
      q[e].x += bx;
      q[e].y += by;
      q[e].z += bz;
    }
  }
  fence_proxy_async_smem();  // before later bulk copies into the same bytes
  __syncwarp();
}

template <bool HALF, int LANES, bool ENERGY, int NB>
__global__ void __launch_bounds__(pipe_threads(NB), 1)
    k_force_pipe(const uint4* __restrict__ pos, Geom g, TileArgs ta, LJConst c, const uint2* __restrict__ rows,
                 const uint2* __restrict__ tile_list, const uint16_t* __restrict__ ent, void* __restrict__ fout,
                 double* __restrict__ part, int32_t* __restrict__ status, const int* __restrict__ skip) {
  constexpr int CW = kPipeConsumers;
  wait_for_previous_launch();
  if (skip && *skip) return;  // a device-decided run stopped before this step
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ PipeTile SS[NB];
  __shared__ __align__(8) uint64_t full[NB], ready[NB], empty[NB];
  const TileLayout L = tile_layout(ta, true, true, false);
  const size_t buf_bytes = align16(L.total);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int b = 0; b < NB; ++b) {
      mbar_init(&full[b], 1);
      mbar_init(&ready[b], 1);
      mbar_init(&empty[b], CW);
    }
    fence_proxy_async_smem();
  }
  __syncthreads();
  EAcc eacc;
  eacc.vscale = g.qu;
  const int64_t stride = gridDim.x;
  const long long budget = wait_budget();
  if (warp >= CW) {
    // ---- producer b: tiles k = b, b + NB, ... in buffer b ----
    const int b = warp - CW;
    unsigned char* buf = smem + b * buf_bytes;
    const uint2* __restrict__ desc = tile_list + ta.ntiles;
    auto load = [&](int64_t t) {
      return lane < kTileDescWords ? desc[kTileDesc * t + lane] : (lane == kTileDescWords ? tile_list[t] : make_uint2(0u, 0u));
    };
    int64_t t = blockIdx.x + b * stride;
    uint2 d = make_uint2(0u, 0u);
    if (t < ta.ntiles) d = load(t);
    uint32_t fills = 0;  // fills of the buffer so far: a phase of full[b] each (a skipped tile has none)
    for (uint32_t use = 0; t < ta.ntiles; t += NB * stride, ++use) {
      const uint32_t total = __shfl_sync(0xffffffffu, d.x, 18), own = __shfl_sync(0xffffffffu, d.y, 18);
      const int gown0 = (int)__shfl_sync(0xffffffffu, d.x, 19), n_own = (int)(own >> 16);
      const bool images = __shfl_sync(0xffffffffu, d.y, 19) != 0u;
      const uint32_t lbase = __shfl_sync(0xffffffffu, d.x, kTileDescWords),
                     llen = __shfl_sync(0xffffffffu, d.y, kTileDescWords);
      bool staged = true;
      if (total > (uint32_t)ta.max_staged) {
        if (lane == 0) atomicOr(status, LJ_ST_CELL_RANGE);
        staged = false;
      } else if (n_own > ta.max_own || llen > (uint32_t)ta.max_list) {
        if (lane == 0) atomicOr(status, LJ_ST_LIST_OVERFLOW);
        staged = false;
      }
      const int r0 = gown0 & ~1, r1 = (gown0 + n_own + 1) & ~1;
      const unsigned n_ent = min(llen, (unsigned)ta.list_cap);  // rows beyond the capacity stay in HBM
      bool ok = true;
      if (use > 0) {
        if (lane == 0) ok = mbar_wait(&empty[b], (use - 1u) & 1u, budget);
        ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
      }
      if (!ok) {  // the consumers did not release the buffer: give up (nothing in flight)
        if (lane == 0) {
          atomicOr(status, LJ_ST_TIMEOUT);
          SS[b].valid = -1;
          mbar_arrive(&ready[b]);
        }
        break;
      }
      if (staged) {
        if (lane == 0) {
          fence_proxy_async_smem();
          mbar_arrive_expect(&full[b], 16u * total + (n_own > 0 ? 8u * (unsigned)(r1 - r0) : 0u) + 2u * n_ent);
        }
        __syncwarp();
        if (lane < 18) {
          const uint32_t n = d.y & 0xffffu;
          if (n > 0) bulk_g2s(buf + L.pos + 16 * (size_t)(d.y >> 16), pos + d.x, 16u * n, &full[b]);
        } else if (lane == 18) {
          if (n_own > 0) bulk_g2s(buf + L.rows, rows + r0, 8u * (unsigned)(r1 - r0), &full[b]);
        } else if (lane == 19) {
          if (n_ent > 0) bulk_g2s(buf + L.ent, ent + lbase, 2u * n_ent, &full[b]);
        } else if (lane == 20) {
          SS[b].own0 = (int)(own & 0xffffu);
          SS[b].own1 = (int)(own & 0xffffu) + n_own;
          SS[b].gown0 = gown0;
          SS[b].row_off = gown0 - r0;
          SS[b].list_base = lbase;
          SS[b].list_len = llen;
        }
      }
      uint32_t ax = 0u, ay = 0u, az = 0u;
      if (staged && images) {
        const uint32_t cxy = __shfl_sync(0xffffffffu, d.x, 20), zt = __shfl_sync(0xffffffffu, d.y, 20);
        const int n = (int)__shfl_sync(0xffffffffu, d.x, 21);
        Geom gs = g;
        gs.Lq = __shfl_sync(0xffffffffu, d.y, 21);
        const TileInfo ti{(int)(cxy & 0xffffu), (int)(cxy >> 16), (int)(zt & 0xffffu), (int)(zt >> 16)};
        if (lane < 18) {
          int sx, sy, sz;
          tile_run_shift(ti, n, lane, sx, sy, sz);
          ax = shift_q(0u, sx, gs);
          ay = shift_q(0u, sy, gs);
          az = shift_q(0u, sz, gs);
        }
      }
      const uint32_t run = lane < 18 ? d.y : 0u;
      const int64_t tn = t + NB * stride;
      if (tn < ta.ntiles) d = load(tn);
      if (staged) {
        bool landed = true;
        if (lane == 0) landed = mbar_wait(&full[b], fills & 1u, budget);
        landed = __shfl_sync(0xffffffffu, landed ? 1 : 0, 0) != 0;
        if (!landed) {
          if (lane == 0) {
            atomicOr(status, LJ_ST_TIMEOUT);
            mbar_wait(&full[b], fills & 1u, kWaitBudget);  // let copies in flight land before leaving
            SS[b].valid = -1;
            mbar_arrive(&ready[b]);
          }
          break;
        }
        ++fills;
        if (images) pipe_shift((uint4*)(buf + L.pos), run, ax, ay, az, lane);
      }
      __syncwarp();
      if (lane == 0) {
        SS[b].valid = staged ? 1 : 0;
        mbar_arrive(&ready[b]);  // release: bookkeeping and copies visible to the consumers
      }
    }
  } else {
    // ---- consumers ----
    // The keys of all of the CTA's tiles in turn, 32 / LANES at a time, go round the consumer warps: a
    // warp without a share of a tile goes on to the next one, so that no warp waits for tiles whose
    // keys do not fill the warps (and the sums stay in a fixed order).
    constexpr int kChunk = 32 / LANES;
    int turn = warp;  // chunk of the current tile that is this warp's next
    int b = 0;
    uint32_t use = 0;  // times the buffer was used before
    for (int64_t t = blockIdx.x; t < ta.ntiles; t += stride) {
      bool ok = __all_sync(0xffffffffu, mbar_wait(&ready[b], use & 1u, budget)) != 0;
      if (!ok) {
        if (lane == 0) atomicOr(status, LJ_ST_TIMEOUT);
        break;
      }
      const PipeTile& S = SS[b];
      if (S.valid < 0) break;
      if (S.valid > 0) {
        const int chunks = (S.own1 - S.own0 + kChunk - 1) / kChunk;
        if (turn < chunks)
          force_tile_compute<true, LANES, HALF, ENERGY, false, true, 32 * CW>(
              S, smem + b * buf_bytes, L, rows, ent, c, g, fout, status, eacc, ta.list_cap, turn * kChunk + lane / LANES);
        turn = (turn - chunks) % CW;
        if (turn < 0) turn += CW;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[b]);
      if (++b == NB) {
        b = 0;
        ++use;
      }
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
// Its launches; all return the grid launched (the number of energy partials written).
template <bool HALF, int LANES, bool ENERGY, int NB>
static int force_pipe_launch(const ForceLaunch& a) {
  const size_t sm = NB * align16(tile_layout(a.ta, true, true, false).total);
  set_smem(k_force_pipe<HALF, LANES, ENERGY, NB>, sm);
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(sm_count(), a.ta.ntiles));
  if (a.overlap)
    launch_overlapping(k_force_pipe<HALF, LANES, ENERGY, NB>, grid, pipe_threads(NB), sm, a.s, (const uint4*)a.pos, a.g,
                       a.ta, a.c, a.rows, a.tile_list, a.ent, a.f, a.part, a.status, a.skip);
  else
    k_force_pipe<HALF, LANES, ENERGY, NB><<<grid, pipe_threads(NB), sm, a.s>>>(
        (const uint4*)a.pos, a.g, a.ta, a.c, a.rows, a.tile_list, a.ent, a.f, a.part, a.status, a.skip);
  return grid;
}
template <bool HALF, int LANES, bool ENERGY>
static int force_pipe(const ForceLaunch& a) {
  switch (a.nbuf) {
    case 2: return force_pipe_launch<HALF, LANES, ENERGY, 2>(a);
    case 3: return force_pipe_launch<HALF, LANES, ENERGY, 3>(a);
    default: return force_pipe_launch<HALF, LANES, ENERGY, 4>(a);
  }
}
template <bool HALF, int LANES>
static int force_pipe_energy(const ForceLaunch& a) {
  return a.energy ? force_pipe<HALF, LANES, true>(a) : force_pipe<HALF, LANES, false>(a);
}

}  // namespace ljmd
