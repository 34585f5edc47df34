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
// Pipelined force (mixed form, full list, tiled box): one CTA per SM, NB producer warps that stage
// tiles into NB shared-memory buffers (producer p handles the tiles k = p mod NB, in buffer p) and 24
// consumer warps that share the keys of all staged tiles, so neither the copies nor the tile-end
// stragglers hold anybody at a barrier.  Per tile k (buffer b = k % NB):
//   producer: wait empty[b] (tile k - NB released) -> issue the copies of tile k from its descriptor
//             (loaded one tile earlier) -> wait full[b] -> (boundary tiles: image shifts) -> arrive ready[b];
//   consumers: wait ready[b] -> forces of the warp's share of the tile's own particles -> arrive
//             empty[b].
// Every wait is bounded; a producer that gives up marks the slot aborted and releases the
// consumers, which then leave.  No copy is in flight when a warp leaves.
//
// Bound by issue (67 % busy) and by the latency of a warp's pair chain, so what counts is that all warps
// always have keys and that the producers, whose dependent instructions each wait their turn among 28
// warps, have little to do.  With a producer working out a tile's cell bounds and prefix sums (40 to 60 %
// of its time), two CTAs of two buffers, a tile's keys spread from the first warp on and scalar pair
// arithmetic, a launch took 2.01 ms at 16.4M particles, rho 0.5 (12 cells per tile), and 78 us at
// 500,000; now 1.32 ms and 55 us.  Packed arithmetic alone gave 1.92 ms, staging the front of long segments
// 1.86 ms, four buffers in one CTA 1.83 ms, the descriptors 1.32 ms.
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

template <int LANES, bool ENERGY, int NB>
__global__ void __launch_bounds__(pipe_threads(NB), 1)
    k_force_pipe(const uint4* __restrict__ pos, Geom g, TileArgs ta, LJConst c, const uint2* __restrict__ rows,
                 const uint2* __restrict__ tile_list, const uint16_t* __restrict__ ent, void* __restrict__ fout,
                 double* __restrict__ part, int32_t* __restrict__ status, const int* __restrict__ skip) {
  constexpr int CW = kPipeConsumers;
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
        if (lane == 0) landed = mbar_wait(&full[b], use & 1u, budget);
        landed = __shfl_sync(0xffffffffu, landed ? 1 : 0, 0) != 0;
        if (!landed) {
          if (lane == 0) {
            atomicOr(status, LJ_ST_TIMEOUT);
            mbar_wait(&full[b], use & 1u, kWaitBudget);  // let copies in flight land before leaving
            SS[b].valid = -1;
            mbar_arrive(&ready[b]);
          }
          break;
        }
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
          force_tile_compute<true, LANES, false, ENERGY, false, true, 32 * CW>(
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
template <int LANES, bool ENERGY, int NB>
static int force_pipe_launch(const ForceLaunch& a) {
  const size_t sm = NB * force_buffer_bytes(a.ta, LJ_MIXED, 0);
  set_smem(k_force_pipe<LANES, ENERGY, NB>, sm);
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(sm_count(), a.ta.ntiles));
  k_force_pipe<LANES, ENERGY, NB><<<grid, pipe_threads(NB), sm, a.s>>>((const uint4*)a.pos, a.g, a.ta, a.c, a.rows,
                                                                       a.tile_list, a.ent, a.f, a.part, a.status, a.skip);
  return grid;
}
template <int LANES, bool ENERGY>
static int force_pipe(const ForceLaunch& a) {
  switch (a.nbuf) {
    case 2: return force_pipe_launch<LANES, ENERGY, 2>(a);
    case 3: return force_pipe_launch<LANES, ENERGY, 3>(a);
    default: return force_pipe_launch<LANES, ENERGY, 4>(a);
  }
}
template <int LANES>
static int force_pipe_energy(const ForceLaunch& a) {
  return a.energy ? force_pipe<LANES, true>(a) : force_pipe<LANES, false>(a);
}

// Buffers of the pipelined kernel for these tiles (0: not even two fit) and the entries of a segment
// that each stages: four, as long as they hold three quarters of the longest segment, else fewer.
static int pipe_plan(TileArgs& ta) {
  int dev = 0, smem_max = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  TileArgs tz = ta;
  tz.list_cap = 0;
  const int64_t fixed = (int64_t)force_buffer_bytes(tz, LJ_MIXED, 0);
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
  } else if (!ta.whole && nbuf == 2 && (a.nbuf = pipe_plan(a.ta)) > 0) {
    switch (lanes) {
      case 1: return force_pipe_energy<1>(a);
      case 2: return force_pipe_energy<2>(a);
      case 4: return force_pipe_energy<4>(a);
      case 8: return force_pipe_energy<8>(a);
      case 16: return force_pipe_energy<16>(a);
      default: return force_pipe_energy<32>(a);
    }
  } else {
    a.nbuf = 1;
    a.smem = force_smem_bytes(ta, precision, 1, half);
    force_tile_mixed<false>(a);
  }
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
        case 2: return force_pipe<2, false>(a);
        case 8: return force_pipe<8, false>(a);
        default: return force_pipe<4, false>(a);
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
