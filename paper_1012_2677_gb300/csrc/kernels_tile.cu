// Cell-column tiles staged in shared memory: pair-list construction (Alg. 1 over the grid of
// Sec. 2.2, stored as the sorted list of Sec. 2.4), tile sizes and list export.  The force over that list
// (Alg. 4-6) and the adjoint pass, which stage the same tiles, have translation units of their own.
//
// A tile is T consecutive cells along z of one (cx, cy) column.  Its CTA stages the particles
// of the 9 neighbouring columns over the cells z0-1 .. z0+T (9 (T+2) cells, wrapped
// periodically) into shared memory.  The cells of one column are contiguous in the cell-sorted
// particle arrays (except where z wraps), so each column is one to three contiguous ranges:
// one lane per column issues asynchronous bulk copies (cp.async.bulk) of those ranges, plus
// the tile's rows and its list segment, all completing on one mbarrier that the CTA waits on
// (bounded).  The periodic image shifts (-L, 0, +L per axis) are then added in shared memory.
//
// Mixed form, force and adjoint kernels: the copies are the fixed-point coordinates of the stored
// FP64 positions (X = round(x / u) mod 2^32, u = 2^-qk, one 16-byte record per particle with the
// sorted index in w), the image shift is the integer round(L / u), and a partner difference is
// the exact integer X_j - X_i converted once to FP32.  List kernels: the FP32 hi parts (top 24
// significand bits) of the stored coordinates, whose differences are exact.  FP64 form: the FP64
// coordinates, the periodic images put in place when staged (one rounding per staged coordinate).
//
// The list holds 16-bit indices into the key particle's staged tile; rows are (start, length)
// per particle; the rows of one tile form one contiguous segment, padded to 8 entries so that
// it can be bulk-copied.  If the box has fewer than 3 cells per side the whole box is one tile
// (all particles staged directly, no shifts, image chosen per pair).
//
// List construction: one lane per key particle tests the three cells around its own in each of
// the 9 neighbour columns (the 27 cells of Alg. 1) from shared memory, FP32 on hi differences,
// which are exact, so r^2 is within a bounded error of the FP64 value; inside that band the FP64
// no-FMA test of the oracle decides, and the pair set equals brute force bit for bit.  The kept
// bits are counted, one atomic per tile reserves the tile's segment, and the entries are written
// from the bits (k_list_win).  The whole-box case (k_list_tile) takes a warp per key particle
// with ballot compaction.
#include "tile.cuh"

namespace ljmd {

template <bool MIXED, bool HALF, bool WHOLE>
__global__ void __launch_bounds__(kTileThreads, 4)
    k_list_tile(const void* __restrict__ pos, const double* __restrict__ x, const uint32_t* __restrict__ cs, int64_t N,
                Geom g, TileArgs ta, ListBand band, uint2* __restrict__ rows, uint2* __restrict__ tile_list,
                uint16_t* __restrict__ ent, uint64_t cap, unsigned long long* __restrict__ counter,
                unsigned int* __restrict__ max_list, int32_t* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ TileShared S;
  __shared__ __align__(8) uint64_t bar;
  __shared__ int s_ok;
  __shared__ unsigned int s_base;
  const TileLayout L = tile_layout(ta, MIXED, false);
  int* sh_gid = (int*)(smem + L.gid);
  int* s_cnt = (int*)(smem + L.cnt);                  // [max_own]
  int* s_pre = s_cnt + ta.max_own;                    // [max_own]
  uint32_t* masks = (uint32_t*)(s_pre + ta.max_own);  // [max_own * max_chunks]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  uint32_t phase = 0;
  if (!WHOLE) {
    if (threadIdx.x == 0) {
      mbar_init(&bar, 1);
      fence_proxy_async_smem();
    }
    __syncthreads();
  }

  for (int64_t t = blockIdx.x; t < ta.ntiles; t += gridDim.x) {
    TileInfo ti{0, 0, 0, 1};
    if (WHOLE) {
      stage_whole<MIXED, true>(N, pos, S, smem, L);
    } else {
      ti = tile_info(t, ta);
      if (!stage_offsets(ti, ta, cs, S)) {
        if (threadIdx.x == 0) atomicOr(status, LJ_ST_CELL_RANGE);
        __syncthreads();
        continue;
      }
      if (!stage_copy_async<MIXED, false>(ti, ta, g, pos, nullptr, nullptr, S, smem, L, &bar, phase, true, status))
        return;
    }
    __syncthreads();
    const int n_own = S.own1 - S.own0;
    const int nk = WHOLE ? 1 : 9;
    if (n_own > ta.max_own) {  // sizing inconsistency: record and skip the tile
      if (threadIdx.x == 0) atomicOr(status, LJ_ST_CELL_RANGE);
      __syncthreads();
      continue;
    }
    // phase 1: test, keep ballots, count
    for (int o = warp; o < n_own; o += kWarps) {
      const int l = S.own0 + o;
      const int gi = sh_gid[l];
      const int m = WHOLE ? 0 : own_cell(S, l, ti.Tp);
      int cnt = 0, c = 0;
      for (int k = 0; k < nk; ++k) {
        const int a = WHOLE ? 0 : S.offq[k * S.ncol + m - 1], b = WHOLE ? S.total : S.offq[k * S.ncol + m + 2];
        for (int base = a; base < b; base += 32) {
          const int j = base + lane;
          bool in = false;
          if (j < b && j != l && (!HALF || sh_gid[j] > gi))
            in = candidate_in<MIXED, WHOLE>(smem, L, l, j, x, N, g, band);
          const unsigned msk = __ballot_sync(0xffffffffu, in);
          if (lane == 0 && c < ta.max_chunks) masks[o * ta.max_chunks + c] = msk;
          ++c;
          cnt += __popc(msk);
        }
      }
      if (lane == 0) s_cnt[o] = (c <= ta.max_chunks) ? cnt : -1;
    }
    __syncthreads();
    if (warp == 0) {
      // exclusive prefix of the row sizes; one atomic reserves the tile's segment, padded to a
      // multiple of 8 entries (16 bytes) so that the force kernel can bulk-copy it
      unsigned run = 0;
      bool ok = true;
      for (int base = 0; base < n_own; base += 32) {
        const int o = base + lane;
        const int v0 = o < n_own ? s_cnt[o] : 0;
        ok = ok && __all_sync(0xffffffffu, v0 >= 0);
        const unsigned v = v0 > 0 ? (unsigned)v0 : 0u;
        unsigned inc = v;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const unsigned y = __shfl_up_sync(0xffffffffu, inc, d);
          if (lane >= d) inc += y;
        }
        if (o < n_own) s_pre[o] = (int)(run + inc - v);
        run += __shfl_sync(0xffffffffu, inc, 31);
      }
      if (lane == 0) {
        const unsigned padded = (run + 7u) & ~7u;
        const unsigned long long b = atomicAdd(counter, (unsigned long long)padded);
        atomicAdd(counter + 1, (unsigned long long)run);
        const bool fits = ok && (b + padded <= cap);
        s_base = (unsigned)b;
        s_ok = fits;
        tile_list[t] = fits ? make_uint2((unsigned)b, padded) : make_uint2(0u, 0u);
        atomicMax(max_list, padded);
        if (!ok) atomicOr(status, LJ_ST_CELL_RANGE);
      }
    }
    __syncthreads();
    // phase 2: rows and entries
    for (int o = warp; o < n_own; o += kWarps) {
      const int l = S.own0 + o;
      const int gi = sh_gid[l];
      const int m = WHOLE ? 0 : own_cell(S, l, ti.Tp);
      const unsigned start = s_base + (unsigned)s_pre[o];
      if (lane == 0) rows[gi] = s_ok ? make_uint2(start, (unsigned)s_cnt[o]) : make_uint2(0u, 0u);
      if (!s_ok) continue;
      unsigned p = start;
      int c = 0;
      for (int k = 0; k < nk; ++k) {
        const int a = WHOLE ? 0 : S.offq[k * S.ncol + m - 1], b = WHOLE ? S.total : S.offq[k * S.ncol + m + 2];
        for (int base = a; base < b; base += 32) {
          const unsigned msk = masks[o * ta.max_chunks + c];
          ++c;
          if ((msk >> lane) & 1u) ent[p + __popc(msk & lt)] = (uint16_t)(base + lane);
          p += __popc(msk);
        }
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------------
// Pair-list construction by cell windows (staged tiles, both forms, both list kinds).
//
// The keys of a tile are taken 32 at a time (a group, one key per lane, consecutive in the cell
// order, so a group spans two or three own cells).  A work item is (group, neighbour column k):
// every lane tests its own key against the three cells m-1, m, m+1 of column k around its own
// cell m (the window of Alg. 1: partners farther along z fail the distance test, cells being at
// least r_s wide).  Lanes in one cell read the same staged record, so a load serves a group with
// one or a few distinct addresses.  The kept-candidate bits of each 32-candidate word go to a
// per-tile pool in shared memory; a count per (key, column) gives every key its row and each
// column its place in the row (columns in order, partners ascending: the list is deterministic);
// one atomic reserves the tile's segment (padded to 8 entries) while the entries are written from
// the bits into shared memory over the staged positions (no longer needed) and then copied out
// with 16-byte stores.  Items whose bits do not fit in the pool are tested again when written (and
// that tile's entries go to global memory directly).  Warp 0 takes the next tile's bookkeeping while
// the others count, its cell bounds copied a tile ahead with cp.async.  With the half list, a
// column other than the key's own has all its cells before or all after the key's in the cell
// order (cell = (X n + Y) n + Z), so such a column is kept or skipped as a whole; in the own column
// the sorted indices decide per pair.
constexpr int kWinPoolPerItem = 2;  // pool words per work item on average (two words hold 64 candidates)
constexpr int kWinThreads = 256;    // threads of a window-kernel CTA
constexpr int kWinCtas = 3;         // window-kernel CTAs resident per SM (register budget)

struct WinLayout {
  size_t pos;    // hi float4 [max_staged + 32] (w: sorted index bits; 32 slack records for the last word);
                 // once the bits are taken, the tile's segment (uint16 [seg_cap]) before it is copied out
  size_t cell;   // uint8 [max_own]: own cell (1..Tp) of each key
  size_t cnt;    // uint16 [ngrp * 9 * 32]: per (key, column) count, then its offset in the key's row
  size_t kst;    // int [max_own]: row start in the segment; then int [max_own]: row length
  size_t ib;     // int [ngrp * 9]: first pool word of each item (-1: tested again when written)
  size_t gtot;   // int [ngrp]: entries of each group of 32 keys
  size_t mask;   // uint32 [pool_words * 32]
  int ngrp, pool_words, seg_cap;
  size_t total;
};

__host__ __device__ __forceinline__ WinLayout win_layout(const TileArgs& ta) {
  WinLayout W;
  const size_t ms = (size_t)ta.max_staged + 32;
  W.ngrp = (ta.max_own + 31) / 32;
  W.pos = 0;
  size_t o = align16(ms * 16);
  W.seg_cap = (int)((ms * 8) & ~(size_t)7);
  W.cell = o;
  o += align16((size_t)ta.max_own);
  W.cnt = o;
  o += align16((size_t)W.ngrp * 9 * 32 * 2);
  W.kst = o;
  o += align16((size_t)ta.max_own * 8);
  W.ib = o;
  o += align16((size_t)W.ngrp * 9 * 4);
  W.gtot = o;
  o += align16((size_t)W.ngrp * 4);
  W.pool_words = W.ngrp * 9 * kWinPoolPerItem + 8;
  W.mask = o;
  o += (size_t)W.pool_words * 32 * 4;
  W.total = o;
  return W;
}

// Order of neighbour column k against the tile's own column, for the half list: +1 if all cells of
// column k come after the tile's own cells in the cell order, -1 if all come before, 0 for the own
// column (decided per pair by the sorted indices).
__device__ __forceinline__ int win_column_order(const TileInfo& ti, int n, int k) {
  if (k == 4) return 0;
  int sx, sy;
  const int X = wrap_cell(ti.cx + k / 3 - 1, n, sx);
  const int Y = wrap_cell(ti.cy + k % 3 - 1, n, sy);
  return (X > ti.cx || (X == ti.cx && Y > ti.cy)) ? 1 : -1;
}

// One 32-candidate word of a key: bit u set iff staged slot jb + u is listed for the key (slot l,
// sorted index gi, hi record pi).  `rem` candidates of the key remain from jb on (the rest of the
// word is masked); lanes without any read slots 0..31 and keep nothing.  Only the first nblk blocks of
// 8 candidates are tested (the windows of all lanes end before the rest).  FP32 filter on the exact
// hi differences; for a word with a kept r^2 inside the band the FP64 test of the oracle decides
// those.  OWN: the key's own column (the key itself is dropped; HALF keeps larger sorted indices).
template <bool HALF, bool OWN>
__device__ __forceinline__ uint32_t win_word(const float4* sh_pos, const double* __restrict__ x, int64_t N,
                                             const Geom& g, const ListBand& band, int jb, int rem, int nblk, int l,
                                             int gi, float4 pi) {
  uint32_t bits = 0;
  float mx = 0.f;
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    if (b >= nblk) break;  // warp-uniform: blocks of 8 past every lane's window are not tested
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const int u = 8 * b + v;
      const float4 pj = sh_pos[jb + u];
      const float dx = pj.x - pi.x, dy = pj.y - pi.y, dz = pj.z - pi.z;  // exact
      const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
      bool in = r2 < band.hi;
      if (HALF && OWN) in = in && __float_as_int(pj.w) > gi;
      if (in) {
        bits |= 1u << u;
        mx = fmaxf(mx, r2);
      }
    }
  }
  bits &= rem >= 32 ? 0xffffffffu : (rem > 0 ? (1u << rem) - 1u : 0u);
  if (OWN) {
    const int d = l - jb;
    if (d >= 0 && d < 32) bits &= ~(1u << d);  // the key itself
  }
  const bool band_hit = bits != 0u && mx >= band.lo;
  if (__any_sync(0xffffffffu, band_hit) && band_hit) {
    uint32_t mb = bits;
    while (mb) {
      const int u = __ffs(mb) - 1;
      mb &= mb - 1;
      const float4 pj = sh_pos[jb + u];
      const float dx = pj.x - pi.x, dy = pj.y - pi.y, dz = pj.z - pi.z;
      const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
      if (r2 >= band.lo && !pair_in_exact(x, N, gi, __float_as_int(pj.w), g, band.rs2)) bits &= ~(1u << u);
    }
  }
  return bits;
}

template <bool HALF>
__device__ __forceinline__ uint32_t win_word_k(bool own, const float4* sh_pos, const double* __restrict__ x,
                                               int64_t N, const Geom& g, const ListBand& band, int jb, int rem,
                                               int nblk, int l, int gi, float4 pi) {
  return own ? win_word<HALF, true>(sh_pos, x, N, g, band, jb, rem, nblk, l, gi, pi)
             : win_word<HALF, false>(sh_pos, x, N, g, band, jb, rem, nblk, l, gi, pi);
}

size_t list_smem_bytes(const TileArgs& ta, int precision) {
  if (!ta.whole) return win_layout(ta).total;  // both forms: the FP32 filter on the hi copies
  return tile_layout(ta, precision == LJ_MIXED, false).total;
}

// DESC: the pipelined force kernel follows, so its staging descriptors are written.
template <bool HALF, bool BATCHED, bool DESC, int NT>
__global__ void __launch_bounds__(NT, kWinCtas)
    k_list_win(const float4* __restrict__ pos, const double* __restrict__ x, const uint32_t* __restrict__ cs_in,
               int64_t N, Geom g_in, TileArgs ta_in, ListBand band, uint2* __restrict__ rows,
               uint2* __restrict__ tile_list, uint16_t* __restrict__ ent, uint64_t cap,
               unsigned long long* __restrict__ counter, unsigned int* __restrict__ max_list,
               int32_t* __restrict__ status, const ReplicaGeo* __restrict__ reps, int R,
               const int* __restrict__ pred, const int32_t* __restrict__ tile_rep) {
  static_assert(NT >= 64, "warp 0 prepares the next tile while the others count");
  if (pred && !*pred) return;  // predicated (batched rebuild inside a graph)
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ TileShared Sb[2];  // bookkeeping of the current tile and of the next one
  __shared__ __align__(8) uint64_t bar;
  __shared__ unsigned int s_base;
  __shared__ int s_fits, s_pool, s_retest;
  __shared__ int s_ready[2];  // the buffer's tile fits the capacities
  constexpr int kNW = NT / 32;
  const WinLayout W = win_layout(ta_in);
  TileLayout L;  // the staging helpers' view: hi records (sorted indices in w)
  L.pos = W.pos;
  L.gid = W.pos;
  L.rows = L.ent = L.cnt = L.total = 0;
  const float4* sh_pos = (const float4*)(smem + W.pos);
  unsigned char* s_cell = smem + W.cell;
  uint16_t* s_cnt = (uint16_t*)(smem + W.cnt);
  int* s_kst = (int*)(smem + W.kst);
  int* s_len = s_kst + ta_in.max_own;
  int* s_ib = (int*)(smem + W.ib);
  int* s_gtot = (int*)(smem + W.gtot);
  uint32_t* s_mask = (uint32_t*)(smem + W.mask);
  uint16_t* s_seg = (uint16_t*)(smem + W.pos);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t phase = 0;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_proxy_async_smem();
  }
  __shared__ uint32_t s_pfa[kMaxCells], s_pfb[kMaxCells];  // cell bounds of the tile being prefetched
  TileInfo pf_ti;  // warp 0: that tile
  auto prefetch = [&](int64_t tp) {  // warp 0: a tile's cell bounds, copied a tile ahead of their use
    TileArgs tap = ta_in;
    Geom gp = g_in;
    const uint32_t* csp = cs_in;
    int64_t tlp = tp;
    if (BATCHED) {
      const ReplicaGeo& rg = reps[tile_rep[tp]];
      replica_view(rg, tap, gp);
      csp = cs_in + rg.cell_base;
      tlp = tp - rg.tile_base;
    }
    pf_ti = tile_info(tlp, tap);
    tile_prefetch_async(pf_ti, tap, csp, s_pfa, s_pfb, lane);
  };
  auto prepare = [&](int b) {  // warp 0: buffer b from the prefetched bounds
    const bool okp = tile_prepare_async(pf_ti, s_pfa, s_pfb, ta_in, Sb[b], lane);
    if (lane == 0) s_ready[b] = (okp && Sb[b].own1 - Sb[b].own0 <= ta_in.max_own) ? 1 : 0;
  };
  if (warp == 0 && blockIdx.x < ta_in.ntiles) {
    prefetch(blockIdx.x);
    prepare(0);
    if (blockIdx.x + gridDim.x < ta_in.ntiles) prefetch(blockIdx.x + gridDim.x);
  }
  __syncthreads();

  int buf = 0;
  for (int64_t t = blockIdx.x; t < ta_in.ntiles; t += gridDim.x, buf ^= 1) {
    TileShared& S = Sb[buf];
    TileArgs ta = ta_in;
    Geom g = g_in;
    int64_t tl = t;
    if (BATCHED) {  // the tile's replica: its box, grid and cells
      const ReplicaGeo& rg = reps[tile_rep[t]];
      replica_view(rg, ta, g);
      tl = t - rg.tile_base;
    }
    const TileInfo ti = tile_info(tl, ta);
    auto prepare_next = [&]() {  // warp 0
      if (t + gridDim.x < ta_in.ntiles) {
        prepare(buf ^ 1);
        if (t + 2 * (int64_t)gridDim.x < ta_in.ntiles) prefetch(t + 2 * (int64_t)gridDim.x);
      }
    };
    if (DESC && warp == kNW - 1)  // the pipelined force kernel's staging descriptor
      tile_desc_write(ti, ta.n, g.Lq, S, s_ready[buf] != 0, tile_list + ta_in.ntiles + kTileDesc * t, lane);
    if (!s_ready[buf]) {  // sizing inconsistency: record and skip the tile
      if (threadIdx.x == 0) atomicOr(status, LJ_ST_CELL_RANGE);
      if (warp == 0) prepare_next();
      __syncthreads();
      continue;
    }
    if (threadIdx.x == 0) {
      s_pool = 0;
      s_retest = 0;
    }
    const int n_own = S.own1 - S.own0, ncol = S.ncol;
    // own cell of every key (ordered before the staged records by the barrier that ends the wait)
    for (int m = 1 + warp; m <= ti.Tp; m += kNW) {
      const int a = S.offq[4 * ncol + m] - S.own0, b = S.offq[4 * ncol + m + 1] - S.own0;
      for (int o = a + lane; o < b; o += 32) s_cell[o] = (unsigned char)m;
    }
    stage_issue<true, false>(ti, ta, pos, nullptr, nullptr, S, smem, L, &bar);
    if (!stage_finish<true, false>(ti, ta, g, S, smem, L, &bar, phase, false, status)) return;
    const int ngrp = (n_own + 31) >> 5, nitem = 9 * ngrp;
    // phase A: the kept-candidate bits of every item, a count per (key, column)
    for (int item = warp; item < nitem; item += kNW) {
      const int gq = item / 9, k = item - 9 * gq;
      const int o = 32 * gq + lane;
      const bool valid = o < n_own;
      const int oc = valid ? o : n_own - 1;
      const int l = S.own0 + oc;
      const float4 pi = sh_pos[l];
      const int gi = __float_as_int(pi.w);
      const int m = s_cell[oc];
      const int j0 = S.offq[k * ncol + m - 1];
      int len = valid ? S.offq[k * ncol + m + 2] - j0 : 0;
      if (HALF && win_column_order(ti, ta.n, k) < 0) len = 0;
      const int maxlen = __reduce_max_sync(0xffffffffu, len);
      const int nw = (maxlen + 31) >> 5;
      int base = 0;
      if (lane == 0) {
        base = nw > 0 ? atomicAdd(&s_pool, nw) : 0;
        if (base + nw > W.pool_words) {
          base = -1;
          s_retest = 1;
        }
        s_ib[item] = base;
      }
      base = __shfl_sync(0xffffffffu, base, 0);
      int cnt = 0;
      for (int w = 0; w < nw; ++w) {
        const int rem = len - 32 * w;
        const uint32_t bits = win_word_k<HALF>(k == 4, sh_pos, x, N, g, band, rem > 0 ? j0 + 32 * w : 0, rem,
                                               (maxlen - 32 * w + 7) >> 3, l, gi, pi);
        if (base >= 0) s_mask[(base + w) * 32 + lane] = bits;
        cnt += __popc(bits);
      }
      s_cnt[item * 32 + lane] = (uint16_t)cnt;
    }
    __syncthreads();
    // phase B (warps 1..): each key's column offsets within its row, its row length and its row's
    // place within its group of 32 keys; the group's entries.  Warp 0 meanwhile takes the next
    // tile's bookkeeping.
    if (warp == 0) prepare_next();
    for (int gq = warp - 1; gq >= 0 && gq < ngrp; gq += kNW - 1) {
      int run = 0;
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        uint16_t* c = s_cnt + (9 * gq + k) * 32 + lane;
        const int v = *c;
        *c = (uint16_t)run;
        run += v;
      }
      const int o = 32 * gq + lane;
      const int v = o < n_own ? run : 0;
      int inc = v;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += y;
      }
      if (o < n_own) {
        s_len[o] = run;
        s_kst[o] = inc - v;
      }
      if (lane == 31) s_gtot[gq] = inc;
    }
    __syncthreads();
    // the tile's entries (every thread); one atomic reserves its segment, padded to 8 entries
    int total = 0;
    for (int gq = 0; gq < ngrp; ++gq) total += s_gtot[gq];
    const unsigned padded = ((unsigned)total + 7u) & ~7u;
    const bool staged = padded <= (unsigned)W.seg_cap && !s_retest;
    if (threadIdx.x == 0) {
      const unsigned long long b = atomicAdd(counter, (unsigned long long)padded);
      atomicAdd(counter + 1, (unsigned long long)total);
      const bool fits = b + padded <= cap;
      s_base = (unsigned)b;
      s_fits = fits;
      tile_list[t] = fits ? make_uint2((unsigned)b, padded) : make_uint2(0u, 0u);
      atomicMax(max_list, padded);
      if (BATCHED && !fits) atomicOr(status, LJ_ST_LIST_OVERFLOW);  // no host retry inside a graph
    }
    // phase D: the entries of every item from its bits (or tested again), in row order; staged
    // over the positions (no longer needed unless an item is tested again) and copied out, or
    // written to global memory directly once the segment's place is known
    auto write_items = [&](auto in_shared) {
      uint16_t* dst = decltype(in_shared)::value ? s_seg : ent + s_base;
      for (int item = warp; item < nitem; item += kNW) {
        const int gq = item / 9, k = item - 9 * gq;
        const int o = 32 * gq + lane;
        const bool valid = o < n_own;
        const int oc = valid ? o : n_own - 1;
        const int m = s_cell[oc];
        const int j0 = S.offq[k * ncol + m - 1];
        int len = valid ? S.offq[k * ncol + m + 2] - j0 : 0;
        if (HALF && win_column_order(ti, ta.n, k) < 0) len = 0;
        int gbase = 0;
        for (int q = 0; q < gq; ++q) gbase += s_gtot[q];
        int p = valid ? gbase + s_kst[o] + s_cnt[item * 32 + lane] : 0;
        const int base = s_ib[item];
        if (base >= 0) {
          for (int w = 0; 32 * w < len; ++w) {
            uint32_t bits = s_mask[(base + w) * 32 + lane];
            while (bits) {
              const int u = __ffs(bits) - 1;
              bits &= bits - 1;
              dst[p++] = (uint16_t)(j0 + 32 * w + u);
            }
          }
        } else if (!decltype(in_shared)::value) {
          const int l = S.own0 + oc;
          const float4 pi = sh_pos[l];
          const int gi = __float_as_int(pi.w);
          const int maxlen = __reduce_max_sync(0xffffffffu, len);
          const int nw = (maxlen + 31) >> 5;
          for (int w = 0; w < nw; ++w) {
            const int rem = len - 32 * w;
            uint32_t bits = win_word_k<HALF>(k == 4, sh_pos, x, N, g, band, rem > 0 ? j0 + 32 * w : 0, rem,
                                             (maxlen - 32 * w + 7) >> 3, l, gi, pi);
            while (bits) {
              const int u = __ffs(bits) - 1;
              bits &= bits - 1;
              dst[p++] = (uint16_t)(j0 + 32 * w + u);
            }
          }
        }
      }
    };
    if (staged) {
      write_items(std::true_type());
      __syncthreads();
    } else {
      __syncthreads();
      if (s_fits) write_items(std::false_type());
    }
    const bool fits = s_fits != 0;
    for (int o = threadIdx.x; o < n_own; o += NT) {
      int gbase = 0;
      for (int q = 0; q < (o >> 5); ++q) gbase += s_gtot[q];
      rows[S.gown0 + o] = fits ? make_uint2(s_base + (unsigned)(gbase + s_kst[o]), (unsigned)s_len[o]) : make_uint2(0u, 0u);
    }
    if (staged && fits) {
      const uint4* src = (const uint4*)s_seg;
      uint4* out = (uint4*)(ent + s_base);
      for (unsigned w = threadIdx.x; w < padded / 8u; w += NT) out[w] = src[w];
    }
    // the positions' bytes were read and written by the generic proxy; the next tile's bulk copies
    // (async proxy) write them
    fence_proxy_async_smem();
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------------
// Largest staged and own counts over the tiles of all replicas.
__global__ void k_tile_sizes_batch(const uint32_t* __restrict__ cs_in, TileArgs caps,
                                   const ReplicaGeo* __restrict__ reps, int R, const int32_t* __restrict__ tile_rep,
                                   unsigned int* __restrict__ out) {
  unsigned int mst = 0, mown = 0;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < caps.ntiles;
       t += (int64_t)gridDim.x * blockDim.x) {
    const ReplicaGeo& rg = reps[tile_rep[t]];
    TileArgs ta = caps;
    Geom g;
    replica_view(rg, ta, g);
    const uint32_t* cs = cs_in + rg.cell_base;
    const TileInfo ti = tile_info(t - rg.tile_base, ta);
    const int ncol = ti.Tp + 2;
    unsigned int tot = 0;
    for (int q = 0; q < 9 * ncol; ++q) {
      int sx, sy, sz;
      const uint32_t cq = cell_of_q(ti, ta.n, ncol, q, sx, sy, sz);
      tot += cs[cq + 1] - cs[cq];
    }
    const uint32_t c0 = ((uint32_t)ti.cx * (uint32_t)ta.n + (uint32_t)ti.cy) * (uint32_t)ta.n + (uint32_t)ti.z0;
    mst = max(mst, tot);
    mown = max(mown, cs[c0 + ti.Tp] - cs[c0]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mst = max(mst, __shfl_xor_sync(0xffffffffu, mst, o));
    mown = max(mown, __shfl_xor_sync(0xffffffffu, mown, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&out[0], mst);
    atomicMax(&out[1], mown);
  }
}

// ---------------------------------------------------------------------------------------------
// Expand the list into (key, partner) sorted-index pairs (for inspection).  The whole-box case
// is a template parameter: no barrier sits under a runtime branch.
template <bool WHOLE>
__global__ void __launch_bounds__(kTileThreads, 4)
    k_list_decode(const uint32_t* __restrict__ cs, int64_t N, TileArgs ta, const uint2* __restrict__ rows,
                  const uint16_t* __restrict__ ent, uint64_t E, uint32_t* __restrict__ out,
                  int32_t* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ TileShared S;
  int* sh_gid = (int*)smem;
  for (int64_t t = blockIdx.x; t < ta.ntiles; t += gridDim.x) {
    if (WHOLE) {
      for (int e = threadIdx.x; e < N; e += blockDim.x) sh_gid[e] = e;
      if (threadIdx.x == 0) {
        S.own0 = 0;
        S.own1 = (int)N;
        S.total = (int)N;
      }
    } else {
      const TileInfo ti = tile_info(t, ta);
      if (!stage_offsets(ti, ta, cs, S)) {
        if (threadIdx.x == 0) atomicOr(status, LJ_ST_CELL_RANGE);
        __syncthreads();
        continue;
      }
      for (int s = threadIdx.x; s < S.total; s += blockDim.x) {
        const int q = slot_cell(S, s);
        sh_gid[s] = S.g0[q] + (s - S.offq[q]);
      }
    }
    __syncthreads();
    for (int l = S.own0 + (int)threadIdx.x / 32; l < S.own1; l += kWarps) {
      const int gi = sh_gid[l];
      const uint2 row = rows[gi];
      if ((uint64_t)row.x + row.y > E) {  // inconsistent row: record and skip
        if ((threadIdx.x & 31) == 0) atomicOr(status, LJ_ST_LIST_OVERFLOW);
        continue;
      }
      for (unsigned e = threadIdx.x & 31; e < row.y; e += 32) {
        const int j = ent[row.x + e];
        const bool ok = j < S.total;
        if (!ok) atomicOr(status, LJ_ST_LIST_OVERFLOW);
        out[2 * (size_t)(row.x + e)] = (uint32_t)gi;
        out[2 * (size_t)(row.x + e) + 1] = ok ? (uint32_t)sh_gid[j] : 0xffffffffu;
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------------
// Sets the budget of the bounded device waits (0: the default).  Synchronises the device.
int set_wait_budget(long long cycles) {
  const long long v = cycles > 0 ? cycles : kWaitBudget;
  if (cudaDeviceSynchronize() != cudaSuccess) return -1;
  if (set_unit_wait_budget(v) || set_wait_budget_force(v) || set_wait_budget_force_half(v) ||
      set_wait_budget_force_dp(v) || set_wait_budget_resident(v) || set_wait_budget_adjoint(v) ||
      set_wait_budget_sort(v))
    return -1;
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : -1;
}

void launch_list_tile(int precision, int half, const void* pos, const float4* hi, const double* x, const uint32_t* cs,
                      int64_t N, Geom g, TileArgs ta, ListBand band, uint2* rows, uint2* tile_list, uint16_t* ent,
                      uint64_t cap, unsigned long long* counter, unsigned int* max_list, int32_t* status,
                      cudaStream_t s, const int* pred, bool descriptors) {
  const size_t sm = list_smem_bytes(ta, precision);
  const int grid = tile_grid(ta, per_sm_for(sm));
#define LJ_LIST_LAUNCH(M, H, W)                                                                                 \
  do {                                                                                                          \
    set_smem(k_list_tile<M, H, W>, sm);                                                                         \
    k_list_tile<M, H, W><<<grid, kTileThreads, sm, s>>>(pos, x, cs, N, g, ta, band, rows, tile_list, ent, cap, \
                                                        counter, max_list, status);                             \
  } while (0)
// tiles, either form: one thread per key on the hi copies (the list is the same), as many CTAs as are resident
#define LJ_WIN_LAUNCH(H, D)                                                                                     \
  do {                                                                                                          \
    set_smem(k_list_win<H, false, D, kWinThreads>, sm);                                                         \
    const int wgrid = tile_grid(ta, resident_per_sm(k_list_win<H, false, D, kWinThreads>, kWinThreads, sm));    \
    k_list_win<H, false, D, kWinThreads><<<wgrid, kWinThreads, sm, s>>>(                                        \
        hi, x, cs, N, g, ta, band, rows, tile_list, ent, cap, counter, max_list, status, nullptr, 0, pred,      \
        nullptr);                                                                                               \
  } while (0)
  const bool mixed = precision == LJ_MIXED;
  if (ta.whole) {
    if (mixed) {
      if (half) LJ_LIST_LAUNCH(true, true, true);
      else LJ_LIST_LAUNCH(true, false, true);
    } else {
      if (half) LJ_LIST_LAUNCH(false, true, true);
      else LJ_LIST_LAUNCH(false, false, true);
    }
  } else if (half) {
    if (descriptors) LJ_WIN_LAUNCH(true, true);
    else LJ_WIN_LAUNCH(true, false);
  } else {
    if (descriptors) LJ_WIN_LAUNCH(false, true);
    else LJ_WIN_LAUNCH(false, false);
  }
#undef LJ_LIST_LAUNCH
#undef LJ_WIN_LAUNCH
}

void launch_list_decode(const uint32_t* cs, int64_t N, TileArgs ta, const uint2* rows, const uint16_t* ent,
                        uint64_t E, uint32_t* out, int32_t* status, cudaStream_t s) {
  const size_t sm = ((4 * (size_t)ta.max_staged) + 15) & ~(size_t)15;
  const int grid = tile_grid(ta, 4);
  if (ta.whole) {
    set_smem(k_list_decode<true>, sm);
    k_list_decode<true><<<grid, kTileThreads, sm, s>>>(cs, N, ta, rows, ent, E, out, status);
  } else {
    set_smem(k_list_decode<false>, sm);
    k_list_decode<false><<<grid, kTileThreads, sm, s>>>(cs, N, ta, rows, ent, E, out, status);
  }
}

// Largest staged count and own count over all tiles (sizes the shared-memory tiles).
__global__ void k_tile_sizes(const uint32_t* __restrict__ cs, TileArgs ta, unsigned int* __restrict__ out) {
  unsigned int mst = 0, mown = 0;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < ta.ntiles;
       t += (int64_t)gridDim.x * blockDim.x) {
    const TileInfo ti = tile_info(t, ta);
    const int ncol = ti.Tp + 2;
    unsigned int tot = 0;
    for (int q = 0; q < 9 * ncol; ++q) {
      int sx, sy, sz;
      const uint32_t cq = cell_of_q(ti, ta.n, ncol, q, sx, sy, sz);
      tot += cs[cq + 1] - cs[cq];
    }
    const uint32_t c0 = ((uint32_t)ti.cx * (uint32_t)ta.n + (uint32_t)ti.cy) * (uint32_t)ta.n + (uint32_t)ti.z0;
    mst = max(mst, tot);
    mown = max(mown, cs[c0 + ti.Tp] - cs[c0]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mst = max(mst, __shfl_xor_sync(0xffffffffu, mst, o));
    mown = max(mown, __shfl_xor_sync(0xffffffffu, mown, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&out[0], mst);
    atomicMax(&out[1], mown);
  }
}

void launch_tile_sizes(const uint32_t* cs, TileArgs ta, unsigned int* out, cudaStream_t s) {
  int64_t b = (ta.ntiles + 255) / 256;
  if (b < 1) b = 1;
  if (b > 4096) b = 4096;
  k_tile_sizes<<<(int)b, 256, 0, s>>>(cs, ta, out);
}

// Largest cell occupancy.
__global__ void k_max_count(const uint32_t* __restrict__ cnt, int64_t n, unsigned int* __restrict__ out) {
  unsigned int m = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    m = max(m, cnt[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

void launch_max_count(const uint32_t* cnt, int64_t n, unsigned int* out, cudaStream_t s) {
  int64_t b = (n + 255) / 256;
  if (b < 1) b = 1;
  if (b > 4096) b = 4096;
  k_max_count<<<(int)b, 256, 0, s>>>(cnt, n, out);
}

// ---- batched replicas -----------------------------------------------------------------------
size_t batch_list_smem_bytes(const TileArgs& caps) { return win_layout(caps).total; }

void launch_tile_sizes_batch(const uint32_t* cs, TileArgs caps, const ReplicaGeo* reps, int R,
                             const int32_t* tile_rep, unsigned int* out, cudaStream_t s) {
  int64_t b = (caps.ntiles + 255) / 256;
  if (b < 1) b = 1;
  if (b > 4096) b = 4096;
  k_tile_sizes_batch<<<(int)b, 256, 0, s>>>(cs, caps, reps, R, tile_rep, out);
}

void launch_list_batch(const float4* hi, const double* x, const uint32_t* cs, int64_t N, Geom g, TileArgs caps,
                       ListBand band, uint2* rows, uint2* tile_list, uint16_t* ent, uint64_t cap,
                       unsigned long long* counter, unsigned int* max_list, int32_t* status, const ReplicaGeo* reps,
                       int R, const int32_t* tile_rep, const int* pred, cudaStream_t s) {
  const size_t sm = win_layout(caps).total;
  set_smem(k_list_win<false, true, true, kWinThreads>, sm);
  const int grid = tile_grid(caps, resident_per_sm(k_list_win<false, true, true, kWinThreads>, kWinThreads, sm));
  k_list_win<false, true, true, kWinThreads><<<grid, kWinThreads, sm, s>>>(hi, x, cs, N, g, caps, band, rows, tile_list, ent,
                                                                     cap, counter, max_list, status, reps, R, pred,
                                                                     tile_rep);
}

// ---- list validity: the large displacement check (LDC) of Alg. 2 -----------------------------
// L_D = { i : |x_i - x_ref_i| > th } with th = margin - (an upper bound of the largest
// displacement); x_ref are the FP64 positions the list was built from.  Indices beyond `cap` are
// counted but not stored.
__global__ void k_ldc_collect(const double* __restrict__ x, const double* __restrict__ xref, int64_t N, double th2,
                              int32_t* __restrict__ list, unsigned int cap, unsigned int* __restrict__ count) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
    const double dx = x[i] - xref[i], dy = x[N + i] - xref[N + i], dz = x[2 * N + i] - xref[2 * N + i];
    if (dx * dx + dy * dy + dz * dz > th2) {
      const unsigned int k = atomicAdd(count, 1u);
      if (k < cap) list[k] = (int32_t)i;
    }
  }
}

// Every pair of L_D: unlisted (the list's own exact FP64 test on the build positions says r >= r_s)
// and now closer than r_c (FP64, with a relative safety of 1e-6) raises *flag.  Block (x, y) takes
// the 16 members 16 x .. 16 x + 15 against the 256 members 256 y + threadIdx.x; pairs a < b only.
constexpr int kLdcRows = 16;
__global__ void __launch_bounds__(256) k_ldc_pairs(const double* __restrict__ x, const double* __restrict__ xref,
                                                   int64_t N, Geom g, const int32_t* __restrict__ list, int m,
                                                   double rs2, double rc2, int* __restrict__ flag) {
  __shared__ double sa[kLdcRows][3];
  __shared__ int ia[kLdcRows];
  const int a0 = blockIdx.x * kLdcRows;
  if (threadIdx.x < kLdcRows) {
    const int a = a0 + threadIdx.x;
    const int i = a < m ? list[a] : 0;
    ia[threadIdx.x] = i;
    for (int k = 0; k < 3; ++k) sa[threadIdx.x][k] = x[k * N + i];
  }
  __syncthreads();
  const int b = blockIdx.y * blockDim.x + threadIdx.x;
  if (b >= m || b <= a0) return;  // some a < b remains only if b > a0
  const int j = list[b];
  const double xj = x[j], yj = x[N + j], zj = x[2 * N + j];
  bool hit = false;
  for (int r = 0; r < kLdcRows; ++r) {
    const int a = a0 + r;
    if (a >= m || a >= b) break;
    double t[3] = {xj - sa[r][0], yj - sa[r][1], zj - sa[r][2]};
    double d2 = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (t[k] > g.half_L) t[k] -= g.L;
      else if (t[k] < -g.half_L) t[k] += g.L;
      d2 += t[k] * t[k];
    }
    if (d2 < rc2 * (1.0 + 1e-6) && !pair_in_exact(xref, N, ia[r], j, g, rs2)) hit = true;
  }
  if (hit) atomicOr(flag, 1);
}

void launch_ldc_collect(const double* x, const double* xref, int64_t N, double th2, int32_t* list, unsigned int cap,
                        unsigned int* count, cudaStream_t s) {
  int64_t b = (N + 255) / 256;
  if (b < 1) b = 1;
  if (b > 65535) b = 65535;
  k_ldc_collect<<<(int)b, 256, 0, s>>>(x, xref, N, th2, list, cap, count);
}
void launch_ldc_pairs(const double* x, const double* xref, int64_t N, Geom g, const int32_t* list, int m, double rs2,
                      double rc2, int* flag, cudaStream_t s) {
  dim3 grid((unsigned)((m + kLdcRows - 1) / kLdcRows), (unsigned)((m + 255) / 256));
  k_ldc_pairs<<<grid, 256, 0, s>>>(x, xref, N, g, list, m, rs2, rc2, flag);
}
}  // namespace ljmd
