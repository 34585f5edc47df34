// Staged cell-column tiles: the bookkeeping, asynchronous staging and pair arithmetic shared by the
// list, force, adjoint and resident-run kernels (kernels_tile.cu has the description of a tile).
#pragma once

#include "common.cuh"

#include <algorithm>

namespace ljmd {

constexpr int kTileThreads = 256;
constexpr int kWarps = kTileThreads / 32;
constexpr int kMaxCells = 9 * (kMaxTileT + 2);

// Budget of the waits for a tile's copies and for the other warps of the pipelined kernel (SM
// clock cycles); the waits that let copies in flight land before a CTA leaves keep kWaitBudget.
// Lowered only by ljmd_set_wait_budget, to drive the timeout paths in tests.
static __device__ long long g_wait_budget = kWaitBudget;  // one per translation unit
__device__ __forceinline__ long long wait_budget() { return g_wait_budget; }
// Sets this translation unit's budget (0 on success).
static inline int set_unit_wait_budget(long long cycles) {
  return cudaMemcpyToSymbol(g_wait_budget, &cycles, sizeof(cycles)) == cudaSuccess ? 0 : -1;
}

struct TileInfo {
  int cx, cy, z0, Tp;
};

__device__ __forceinline__ TileInfo tile_info(int64_t t64, const TileArgs& ta) {
  TileInfo ti;
  const unsigned t = (unsigned)t64;  // tiles < 2^31 (n <= 1024)
  const unsigned tz = t % (unsigned)ta.ntz;
  const unsigned r = t / (unsigned)ta.ntz;
  ti.cy = (int)(r % (unsigned)ta.n);
  ti.cx = (int)(r / (unsigned)ta.n);
  ti.z0 = (int)tz * ta.T;
  ti.Tp = min(ta.T, ta.n - ti.z0);
  return ti;
}

// Shared bookkeeping of one staged tile.
struct TileShared {
  int offq[kMaxCells + 1];  // staged index of the first particle of cell q = k (Tp+2) + m
  int g0[kMaxCells];        // sorted (global) index of the first particle of cell q
  int ncol, ncell, total;   // cells per column, staged cells, staged particles
  int own0, own1;           // staged range of the tile's own particles
  int gown0;                // sorted index of the first own particle
  unsigned list_base, list_len;  // the tile's (padded) list segment
  int row_off;              // index of the first own row in the staged row copy
};

// Wrapped coordinate and image shift (-1, 0, +1) of a neighbour cell index.
__device__ __forceinline__ int wrap_cell(int c, int n, int& shift) {
  shift = 0;
  if (c < 0) {
    c += n;
    shift = -1;
  } else if (c >= n) {
    c -= n;
    shift = 1;
  }
  return c;
}

__device__ __forceinline__ uint32_t cell_of_q(const TileInfo& ti, int n, int ncol, int q, int& sx, int& sy, int& sz) {
  const int k = q / ncol, m = q - (q / ncol) * ncol;
  const int X = wrap_cell(ti.cx + k / 3 - 1, n, sx);
  const int Y = wrap_cell(ti.cy + k % 3 - 1, n, sy);
  const int Z = wrap_cell(ti.z0 - 1 + m, n, sz);
  return ((uint32_t)X * (uint32_t)n + (uint32_t)Y) * (uint32_t)n + (uint32_t)Z;
}

// Cell bounds of the tile's 9 (Tp + 2) staged cells and their prefix (one warp).  Returns false
// (all threads) if the tile exceeds the staged capacity.
__device__ __forceinline__ bool stage_offsets(const TileInfo& ti, const TileArgs& ta, const uint32_t* __restrict__ cs,
                                              TileShared& S) {
  const int ncol = ti.Tp + 2;
  const int ncell = 9 * ncol;
  for (int q = threadIdx.x; q < ncell; q += blockDim.x) {
    int sx, sy, sz;
    const uint32_t c = cell_of_q(ti, ta.n, ncol, q, sx, sy, sz);
    const uint32_t a = cs[c], b = cs[c + 1];
    S.g0[q] = (int)a;
    S.offq[q + 1] = (int)(b - a);
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    int run = 0;
    for (int base = 0; base < ncell; base += 32) {
      const int q = base + lane;
      const int v = q < ncell ? S.offq[q + 1] : 0;
      int inc = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      if (q < ncell) S.offq[q + 1] = run + inc;
      run += __shfl_sync(0xffffffffu, inc, 31);
    }
    __syncwarp();
    if (lane == 0) {
      S.offq[0] = 0;
      S.ncol = ncol;
      S.ncell = ncell;
      S.total = run;
      S.own0 = S.offq[4 * ncol + 1];
      S.own1 = S.offq[4 * ncol + ti.Tp + 1];
      S.gown0 = S.g0[4 * ncol + 1];
    }
  }
  __syncthreads();
  return S.total <= ta.max_staged;
}

// Staging descriptor of a tile, kTileDesc words of 8 bytes written by the list kernel where the pipelined force
// kernel follows (behind the tiles' list segments: tile_list + ntiles), which reads one word per lane, so that
// staging a tile takes no bookkeeping at all in the ten or so steps of a list's life:
//   0..17  run 2 k + r of column k: first sorted index; staged slot << 16 | particles (a column is one
//          run, or two where z wraps)
//   18     staged particles (kTileInvalid: the tile exceeded the capacities); own slot | own particles << 16
//   19     sorted index of the first own particle; 1 if the tile has periodic images
//   20     cx | cy << 16; z0 | cells << 16
//   21     cells per side; image shift round(L / u)
constexpr int kTileDesc = kTileWords - 1;
constexpr int kTileDescWords = 22;
constexpr uint32_t kTileInvalid = 0xffffffffu;

__device__ __forceinline__ bool tile_interior(const TileInfo& ti, int n) {
  return ti.cx >= 1 && ti.cx <= n - 2 && ti.cy >= 1 && ti.cy <= n - 2 && ti.z0 >= 1 && ti.z0 + ti.Tp <= n - 1;
}

// The first cell of run r = 1 of a tile's columns (ncol: there is none).
__device__ __forceinline__ int tile_run_cut(int z0, int Tp, int n) {
  return z0 == 0 ? 1 : (z0 + Tp == n ? Tp + 1 : Tp + 2);
}

// Image shifts of run l of a tile.
__device__ __forceinline__ void tile_run_shift(const TileInfo& ti, int n, int l, int& sx, int& sy, int& sz) {
  const int k = l >> 1, r = l & 1;
  wrap_cell(ti.cx + k / 3 - 1, n, sx);
  wrap_cell(ti.cy + k % 3 - 1, n, sy);
  sz = ti.z0 == 0 && r == 0 ? -1 : (ti.z0 + ti.Tp == n && r == 1 ? 1 : 0);
}

// One warp writes the descriptor of a tile from its bookkeeping.
__device__ __forceinline__ void tile_desc_write(const TileInfo& ti, int n, uint32_t Lq, const TileShared& S, bool valid,
                                                uint2* __restrict__ desc, int lane) {
  uint2 d = make_uint2(0u, 0u);
  if (lane < 18) {
    const int k = lane >> 1, r = lane & 1, ncol = S.ncol, cut = tile_run_cut(ti.z0, ti.Tp, n);
    const int m0 = r ? cut : 0, m1 = r ? ncol : cut;
    if (valid && m1 > m0) {
      const int a = S.offq[k * ncol + m0], b = S.offq[k * ncol + m1];
      d = make_uint2((uint32_t)S.g0[k * ncol + m0], (uint32_t)a << 16 | (uint32_t)(b - a));
    }
  } else if (lane == 18) {
    d = make_uint2(valid ? (uint32_t)S.total : kTileInvalid, (uint32_t)S.own0 | (uint32_t)(S.own1 - S.own0) << 16);
  } else if (lane == 19) {
    d = make_uint2((uint32_t)S.gown0, tile_interior(ti, n) ? 0u : 1u);
  } else if (lane == 20) {
    d = make_uint2((uint32_t)(ti.cx | ti.cy << 16), (uint32_t)(ti.z0 | ti.Tp << 16));
  } else if (lane == 21) {
    d = make_uint2((uint32_t)n, Lq);
  }
  if (lane < kTileDescWords) desc[lane] = d;
}

// Cell bounds of a tile's staged cells copied asynchronously into shared memory (one warp; lane m
// takes cell m of every column).  Nothing waits for the loads until tile_prepare_async.
__device__ __forceinline__ void tile_prefetch_async(const TileInfo& ti, const TileArgs& ta,
                                                    const uint32_t* __restrict__ cs, uint32_t* pa, uint32_t* pb,
                                                    int lane) {
  const int ncol = ti.Tp + 2;
  if (lane >= ncol) return;
  int sz;
  const uint32_t Z = (uint32_t)wrap_cell(ti.z0 - 1 + lane, ta.n, sz);
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    int sx, sy;
    const uint32_t X = (uint32_t)wrap_cell(ti.cx + k / 3 - 1, ta.n, sx);
    const uint32_t Y = (uint32_t)wrap_cell(ti.cy + k % 3 - 1, ta.n, sy);
    const uint32_t c = (X * (uint32_t)ta.n + Y) * (uint32_t)ta.n + Z;
    cp_async4(pa + k * ncol + lane, cs + c);
    cp_async4(pb + k * ncol + lane, cs + c + 1);
  }
}

// The bookkeeping of stage_offsets done by one warp from the bounds of tile_prefetch_async.
__device__ __forceinline__ bool tile_prepare_async(const TileInfo& ti, const uint32_t* pa, const uint32_t* pb,
                                                   const TileArgs& ta, TileShared& S, int lane) {
  cp_async_wait_all();
  __syncwarp();
  const int ncol = ti.Tp + 2, ncell = 9 * ncol;
  int run = 0;
  for (int base = 0; base < ncell; base += 32) {
    const int q = base + lane;
    int inc = 0;
    if (q < ncell) {
      const uint32_t a = pa[q];
      inc = (int)(pb[q] - a);
      S.g0[q] = (int)a;
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (q < ncell) S.offq[q + 1] = run + inc;
    run += __shfl_sync(0xffffffffu, inc, 31);
  }
  __syncwarp();  // the bounds are read before the next prefetch overwrites them
  if (lane == 0) {
    S.offq[0] = 0;
    S.ncol = ncol;
    S.ncell = ncell;
    S.total = run;
    S.own0 = S.offq[4 * ncol + 1];
    S.own1 = S.offq[4 * ncol + ti.Tp + 1];
    S.gown0 = S.g0[4 * ncol + 1];
    S.list_base = 0;
    S.list_len = 0;
  }
  __syncwarp();
  return run <= ta.max_staged;
}

// Staged cell of staged slot s: the largest q with offq[q] <= s.
__device__ __forceinline__ int slot_cell(const TileShared& S, int s) {
  int lo = 0, hi = S.ncell - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (S.offq[mid] <= s) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Shared-memory layout of a staged tile (byte offsets from the dynamic shared base).
struct TileLayout {
  size_t pos;    // MIXED: fixed-point uint4 [ms] (force, adjoint) or hi float4 [ms] (list); FP64: dvec4 [ms]
  size_t gid;    // int [ms] (where the sorted index is not carried in the staged record)
  size_t rows;   // uint2 [max_own + 2] (force only)
  size_t ent;    // uint16 [list_cap] (force only)
  size_t cnt;    // int [max_own] (list only), then pre [max_own], then masks [max_own * max_chunks]
  size_t total;
};

static __host__ __device__ __forceinline__ size_t align16(size_t b) { return (b + 15) & ~(size_t)15; }

__host__ __device__ __forceinline__ TileLayout tile_layout(const TileArgs& ta, bool mixed, bool force,
                                                           bool gid = true) {
  TileLayout L;
  const size_t ms = (size_t)ta.max_staged;
  L.pos = 0;
  size_t o = align16(ms * (mixed ? 16 : 32));
  L.gid = o;
  if (gid) o += align16(ms * 4);  // the full-list force kernel needs no sorted indices
  L.rows = o;
  L.ent = o;
  L.cnt = o;
  if (force) {
    o += align16(8 * ((size_t)ta.max_own + 2));
    L.ent = o;
    if (!ta.whole) o += align16(2 * (size_t)ta.list_cap);
  } else {
    o += align16(8 * (size_t)ta.max_own + 4 * (size_t)ta.max_own * ta.max_chunks);
  }
  L.total = o;
  return L;
}

// Issue the bulk copies of one tile (warp 0; lane k < 9 handles column k, lane 9 the rows
// and list segment), all completing on `bar`.  Copies: positions (fixed-point records, hi or FP64), and for the
// force kernel the own rows and the list segment.  No barrier inside: the other warps go on.
template <bool MIXED, bool FORCE>
__device__ __forceinline__ void stage_issue(const TileInfo& ti, const TileArgs& ta, const void* __restrict__ pos,
                                            const uint2* __restrict__ rows, const uint16_t* __restrict__ ent,
                                            TileShared& S, unsigned char* smem, const TileLayout& L, uint64_t* bar) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned bpp = MIXED ? 16u : 32u;
  if (warp != 0) return;
  unsigned bytes = (unsigned)S.total * bpp;
  int r0 = 0, r1 = 0;
  const int n_own = S.own1 - S.own0;
  if (FORCE) {
    r0 = S.gown0 & ~1;
    r1 = (S.gown0 + n_own + 1) & ~1;
    if (n_own > 0) bytes += 8u * (unsigned)(r1 - r0);
    bytes += 2u * min(S.list_len, (unsigned)ta.list_cap);
  }
  if (lane == 0) {
    fence_proxy_async_smem();
    mbar_arrive_expect(bar, bytes);
  }
  __syncwarp();
  if (lane < 9) {
    // column `lane`: cells z0-1 .. z0+Tp wrapped in z; they are contiguous in the sorted arrays
    // except where z wraps (first cell when z0 = 0, last cell when z0 + Tp = n), so one to two runs
    const int k = lane, ncol = S.ncol;
    int cut0 = 0, cut1 = ncol;  // middle run [cut0, cut1); wrapped single cells outside it
    if (ti.z0 == 0) cut0 = 1;
    if (ti.z0 + ti.Tp == ta.n) cut1 = ncol - 1;
    const int bounds[4] = {0, cut0, cut1, ncol};
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int m0 = bounds[r], m1 = bounds[r + 1];
      if (m1 <= m0) continue;
      const int q0 = k * ncol + m0;
      const unsigned n = (unsigned)(S.offq[k * ncol + m1] - S.offq[q0]);
      if (n > 0) {
        const size_t gsrc = (size_t)S.g0[q0];
        const size_t dst = (size_t)S.offq[q0];
        if (MIXED) {
          bulk_g2s(smem + L.pos + 16 * dst, (const uint4*)pos + gsrc, 16u * n, bar);
        } else {
          bulk_g2s(smem + L.pos + 32 * dst, (const dvec4*)pos + gsrc, 32u * n, bar);
        }
      }
    }
  } else if (FORCE && lane == 9) {
    if (n_own > 0) bulk_g2s(smem + L.rows, rows + r0, 8u * (unsigned)(r1 - r0), bar);
    const unsigned n_ent = min(S.list_len, (unsigned)ta.list_cap);  // rows beyond the capacity stay in HBM
    if (n_ent > 0) bulk_g2s(smem + L.ent, ent + S.list_base, 2u * n_ent, bar);
    S.row_off = S.gown0 - r0;
  }
}

// Image shift of one staged fixed-point coordinate by s L (s = -1, 0, +1): the integer s round(L / u)
// added modulo 2^32 (exact; the image carries the rounding of L / u, at most u / 2).
__device__ __forceinline__ uint32_t shift_q(uint32_t q, int s, const Geom& g) {
  return s > 0 ? q + g.Lq : (s < 0 ? q - g.Lq : q);
}

// Wait (all threads, bounded) for the copies of a staged tile, then fill in the image shifts
// (mixed: added to the fixed-point record or to hi; FP64: s L added to the coordinates) and, if
// wanted, the sorted indices.  Returns false
// (all threads) on timeout, after recording it; the caller drains any other copies in flight.
template <bool MIXED, bool FORCE>
__device__ __forceinline__ bool stage_finish(const TileInfo& ti, const TileArgs& ta, const Geom& g, TileShared& S,
                                             unsigned char* smem, const TileLayout& L, uint64_t* bar,
                                             uint32_t& phase, bool want_gid, int32_t* status) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // one thread polls the barrier; the others wait at the CTA barrier without taking issue slots
  bool ok = true;
  if (threadIdx.x == 0) ok = mbar_wait(bar, phase, wait_budget());
  ok = __syncthreads_and(ok) != 0;
  if (!ok) {
    if (threadIdx.x == 0) {
      atomicOr(status, LJ_ST_TIMEOUT);
      mbar_wait(bar, phase, kWaitBudget);  // let copies in flight land before the CTA leaves
    }
    __syncthreads();
    return false;
  }
  phase ^= 1u;
  // interior tiles (no periodic image among the staged cells) need no shifts
  const bool interior = ti.cx >= 1 && ti.cx <= ta.n - 2 && ti.cy >= 1 && ti.cy <= ta.n - 2 && ti.z0 >= 1 &&
                        ti.z0 + ti.Tp <= ta.n - 1;
  if (interior && !want_gid) return true;
  for (int q = warp; q < S.ncell; q += (int)(blockDim.x >> 5)) {
    int sx = 0, sy = 0, sz = 0;
    if (!interior) cell_of_q(ti, ta.n, S.ncol, q, sx, sy, sz);
    const bool shifted = (sx | sy | sz) != 0;
    if (!shifted && !want_gid) continue;
    const int a = S.offq[q], b = S.offq[q + 1], gq = S.g0[q];
    for (int s = a + lane; s < b; s += 32) {
      if (MIXED) {
        if (shifted) {
          if (FORCE) {
            uint4* q = (uint4*)(smem + L.pos) + s;
            q->x = shift_q(q->x, sx, g);
            q->y = shift_q(q->y, sy, g);
            q->z = shift_q(q->z, sz, g);
          } else {  // list filter: hi only; a rounding of hi stays inside the FP32 band
            float4* h = (float4*)(smem + L.pos) + s;
            h->x = fmaf((float)sx, g.L_hi, h->x);
            h->y = fmaf((float)sy, g.L_hi, h->y);
            h->z = fmaf((float)sz, g.L_hi, h->z);
          }
        }
      } else if (shifted) {  // the image itself: one rounding per staged coordinate, none per pair
        dvec4* p = (dvec4*)(smem + L.pos) + s;
        p->x += (double)sx * g.L;
        p->y += (double)sy * g.L;
        p->z += (double)sz * g.L;
      }
      if (want_gid) ((int*)(smem + L.gid))[s] = gq + (s - a);
    }
  }
  // these generic writes precede later bulk copies into the same bytes
  fence_proxy_async_smem();
  __syncthreads();
  return true;
}

// Issue, wait and fix up one tile (single-buffered use).
template <bool MIXED, bool FORCE>
__device__ __forceinline__ bool stage_copy_async(const TileInfo& ti, const TileArgs& ta, const Geom& g,
                                                 const void* __restrict__ pos, const uint2* __restrict__ rows,
                                                 const uint16_t* __restrict__ ent, TileShared& S, unsigned char* smem,
                                                 const TileLayout& L, uint64_t* bar, uint32_t& phase, bool want_gid,
                                                 int32_t* status) {
  stage_issue<MIXED, FORCE>(ti, ta, pos, rows, ent, S, smem, L, bar);
  return stage_finish<MIXED, FORCE>(ti, ta, g, S, smem, L, bar, phase, want_gid, status);
}

// Whole box as one tile (fewer than 3 cells per side): everything staged directly, no shifts.
// GID: also the sorted indices (every layout but the mixed force and adjoint kernels', whose
// fixed-point records carry them).
template <bool MIXED, bool GID>
__device__ __forceinline__ void stage_whole(int64_t N, const void* __restrict__ pos, TileShared& S,
                                            unsigned char* smem, const TileLayout& L) {
  for (int e = threadIdx.x; e < N; e += blockDim.x) {
    if (MIXED) {
      ((uint4*)(smem + L.pos))[e] = ((const uint4*)pos)[e];
    } else {
      dvec4 p = ((const dvec4*)pos)[e];
      p.w = 13.0;  // no shift
      ((dvec4*)(smem + L.pos))[e] = p;
    }
    if (GID) ((int*)(smem + L.gid))[e] = e;
  }
  if (threadIdx.x == 0) {
    S.ncol = 1;
    S.ncell = 1;
    S.total = (int)N;
    S.own0 = 0;
    S.own1 = (int)N;
    S.gown0 = 0;
    S.offq[0] = 0;
    S.offq[1] = (int)N;
  }
}

// Exact list test of the oracle (FP64, fixed min-image formula, no FMA) on stored coordinates.
__device__ __forceinline__ bool pair_in_exact(const double* __restrict__ x, int64_t N, int i, int j, const Geom& g,
                                              double rs2) {
  double d[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double t = __dsub_rn(x[k * N + j], x[k * N + i]);
    if (t > g.half_L) t = __dsub_rn(t, g.L);
    else if (t < -g.half_L) t = __dadd_rn(t, g.L);
    d[k] = t;
  }
  const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
  return r2 < rs2;
}

// Candidate test in FP32 on staged copies (exact hi differences for the mixed form; the FP64
// form rounds its exact difference), then the exact FP64 test inside the band.
template <bool MIXED, bool WHOLE>
__device__ __forceinline__ bool candidate_in(const unsigned char* smem, const TileLayout& L, int li, int lj,
                                             const double* __restrict__ x, int64_t N, const Geom& g,
                                             const ListBand& band) {
  float r2;
  if (MIXED) {
    const float4 a = ((const float4*)(smem + L.pos))[li], b = ((const float4*)(smem + L.pos))[lj];
    float dx = b.x - a.x, dy = b.y - a.y, dz = b.z - a.z;  // exact
    if (WHOLE) {
      dx = fmaf(-rintf(dx * g.inv_L), g.L_hi, dx);
      dy = fmaf(-rintf(dy * g.inv_L), g.L_hi, dy);
      dz = fmaf(-rintf(dz * g.inv_L), g.L_hi, dz);
    }
    r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
  } else {
    const dvec4 a = ((const dvec4*)(smem + L.pos))[li], b = ((const dvec4*)(smem + L.pos))[lj];
    double dx = b.x - a.x, dy = b.y - a.y, dz = b.z - a.z;  // staged tiles: images already in place
    if (WHOLE) {
      dx = fma(-rint(dx * g.inv_L64), g.L, dx);
      dy = fma(-rint(dy * g.inv_L64), g.L, dy);
      dz = fma(-rint(dz * g.inv_L64), g.L, dz);
    }
    const float fx = (float)dx, fy = (float)dy, fz = (float)dz;
    r2 = fmaf(fx, fx, fmaf(fy, fy, fz * fz));
  }
  if (r2 < band.lo) return true;
  if (r2 >= band.hi) return false;
  const int* gid = (const int*)(smem + L.gid);
  return pair_in_exact(x, N, gid[li], gid[lj], g, band.rs2);
}

__device__ __forceinline__ int own_cell(const TileShared& S, int l, int Tp) {
  const int base = 4 * S.ncol;
  int m = 1;
  while (m < Tp && l >= S.offq[base + m + 1]) ++m;
  return m;
}

// ---------------------------------------------------------------------------------------------
// Batched replicas: the tile geometry of a replica (capacities stay the batch's).
__device__ __forceinline__ void replica_view(const ReplicaGeo& rg, TileArgs& ta, Geom& g) {
  ta.n = rg.n;
  ta.T = rg.T;
  ta.ntz = rg.ntz;
  ta.whole = 0;
  ta.ntiles = (int64_t)rg.n * rg.n * rg.ntz;
  g = rg.g;
}

template <int LANES>
__device__ __forceinline__ float gsum(float v) {
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
template <int LANES>
__device__ __forceinline__ double gsum(double v) {
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 1/x from the hardware approximation (rcp.approx) refined by one Newton-Raphson step
// r' = r + r (1 - x r), which roughly squares its relative error.
__device__ __forceinline__ float rcp_nr(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return fmaf(r, fmaf(-x, r, 1.0f), r);
}

// 1/x in FP64 from the hardware approximation (rcp.approx.ftz.f64) refined by two Newton-Raphson
// steps r' = r + r (1 - x r), each of which squares the relative error: full double precision to
// within an ulp, in a handful of FP64 operations instead of a correctly rounded reciprocal.
__device__ __forceinline__ double rcp_nr64(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

// A key's sums over the two pairs a lane takes side by side (x: even, y: odd entries of the lane).
struct AccF {
  float2 fx, fy, fz, pe, vir;
};

// Per-thread energy and virial sums over the keys a thread finishes: FP32 partials of at most
// 16 keys, folded into FP64 totals (so the FP64 pipe, 1/64 of the FP32 rate on this part, sees one
// add per 16 keys).  The mixed form's virial partial is in units of 1/u and is scaled by u
// (exactly: u = 2^-qk) when folded.
struct EAcc {
  double pe = 0.0, vir = 0.0;
  float pe32 = 0.0f, vir32 = 0.0f;
  int n = 0;
  float vscale = 1.0f;
  __device__ __forceinline__ void flush() {
    pe += f32_to_f64(pe32);
    vir += f32_to_f64(vir32 * vscale);
    pe32 = vir32 = 0.0f;
    n = 0;
  }
  __device__ __forceinline__ void add32(float p, float v) {
    pe32 += p;
    vir32 += v;
    if (++n == 16) flush();  // (as a branch: predicated, its FP64 adds would take their slots every time)
  }
};

// Partner difference of two fixed-point records in units of u: the exact integer difference
// converted once to FP32.  WHOLE: the nearest periodic image is chosen per pair (the raw
// difference is below 2^31 u there) and round(L / u) subtracted as an integer.
template <bool WHOLE>
__device__ __forceinline__ float qd(uint32_t a, uint32_t b, const Geom& g) {
  int d = (int)(a - b);
  if (WHOLE) d -= (int)rintf(__int2float_rn(d) * g.q_inv_L) * (int)g.Lq;
  return __int2float_rn(d);
}

// Two listed pairs of one key in the mixed form (Alg. 6 in eps/sigma form) on differences in units of u:
//   f = ri2 s3i (24 eps - 48 eps s3i) + 8 eps c2 / sigma^2, zero for r^2 >= r_c^2 (select)
//   V = 4 eps [s3i (s3i - 1) + c2 r^2 / sigma^2 + c0],  W += -f r^2
// with the constants scaled by powers of u (LJConst::*q), so f d and V come out in sigma units and
// W in units of 1/u.  The FP32 arithmetic is packed two by two (the kernels are bound by issue: one
// packed instruction in the place of two): the reciprocal is taken of -r^2, which keeps every sign out of
// the packed instructions (they have no negation), and the factor 4 eps of V is left to the caller;
// a.vir sums +f r^2.  HALF: d is x_i - x_j, so that f d is the force on the partner, added to its sorted
// index (carried in q.w); a then holds minus the key's sums.  two: the second pair exists (else it
// repeats the first and counts nothing).
template <bool HALF, bool ENERGY, bool WHOLE>
__device__ __forceinline__ void pair2_q(const uint4& qi, const uint4& q0, const uint4& q1, bool two, const LJConst& c,
                                        const Geom& g, AccF& a, float4* fout) {
  float2 dx, dy, dz;
  if (HALF) {
    dx = make_float2(qd<WHOLE>(qi.x, q0.x, g), qd<WHOLE>(qi.x, q1.x, g));
    dy = make_float2(qd<WHOLE>(qi.y, q0.y, g), qd<WHOLE>(qi.y, q1.y, g));
    dz = make_float2(qd<WHOLE>(qi.z, q0.z, g), qd<WHOLE>(qi.z, q1.z, g));
  } else {
    dx = make_float2(qd<WHOLE>(q0.x, qi.x, g), qd<WHOLE>(q1.x, qi.x, g));
    dy = make_float2(qd<WHOLE>(q0.y, qi.y, g), qd<WHOLE>(q1.y, qi.y, g));
    dz = make_float2(qd<WHOLE>(q0.z, qi.z, g), qd<WHOLE>(q1.z, qi.z, g));
  }
  const float2 one = make_float2(1.0f, 1.0f);
  const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
  // -1/r^2: the hardware approximation of it, refined by one Newton-Raphson step (as rcp_nr)
  float2 nr;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(nr.x) : "f"(-r2.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(nr.y) : "f"(-r2.y));
  nr = __ffma2_rn(nr, __ffma2_rn(r2, nr, one), nr);
  const float2 ns = __fmul2_rn(make_float2(c.sig2q, c.sig2q), nr);
  const float2 ns3 = __fmul2_rn(__fmul2_rn(ns, ns), ns);  // -s3i
  float2 ff = __ffma2_rn(__fmul2_rn(nr, ns3), __ffma2_rn(make_float2(c.f48q, c.f48q), ns3, make_float2(c.f24q, c.f24q)),
                         make_float2(c.f8c2q, c.f8c2q));
  const bool in0 = r2.x < c.rc2q, in1 = two && r2.y < c.rc2q;
  ff.x = in0 ? ff.x : 0.0f;
  ff.y = in1 ? ff.y : 0.0f;
  a.fx = __ffma2_rn(ff, dx, a.fx);
  a.fy = __ffma2_rn(ff, dy, a.fy);
  a.fz = __ffma2_rn(ff, dz, a.fz);
  if (HALF) {
    const float2 fx = __fmul2_rn(ff, dx), fy = __fmul2_rn(ff, dy), fz = __fmul2_rn(ff, dz);
    if (in0) atomicAdd(&fout[q0.w], make_float4(fx.x, fy.x, fz.x, 0.0f));
    if (in1) atomicAdd(&fout[q1.w], make_float4(fx.y, fy.y, fz.y, 0.0f));
  }
  if (ENERGY) {
    float2 v = __ffma2_rn(ns3, __fadd2_rn(ns3, one),
                          __ffma2_rn(make_float2(c.c2q, c.c2q), r2, make_float2(c.c0f, c.c0f)));
    v.x = in0 ? v.x : 0.0f;
    v.y = in1 ? v.y : 0.0f;
    a.pe = __fadd2_rn(a.pe, v);
    a.vir = __ffma2_rn(ff, r2, a.vir);
  }
}

// Forces of the own particles of one staged tile (buffer `buf`); LANES threads per key particle, striding
// over its row; a thread's group starts at key grp and steps by the number of groups.
template <bool MIXED, int LANES, bool HALF, bool ENERGY, bool WHOLE, bool LONGLIST, int NTH = kTileThreads, class TS>
__device__ __forceinline__ void force_tile_compute(const TS& S, const unsigned char* buf, const TileLayout& L,
                                                   const uint2* __restrict__ rows, const uint16_t* __restrict__ ent,
                                                   const LJConst& c, const Geom& g, void* __restrict__ fout,
                                                   int32_t* __restrict__ status, EAcc& eacc, int list_cap,
                                                   int grp = threadIdx.x / LANES) {
  const void* sh_pos = buf + L.pos;
  const int* sh_gid = (const int*)(buf + L.gid);
  const uint2* s_rows = (const uint2*)(buf + L.rows);
  const uint16_t* s_ent = (const uint16_t*)(buf + L.ent);
  const int lane = threadIdx.x & (LANES - 1);
  constexpr int kGroups = NTH / LANES;  // groups of the computing threads
  const double f24d = 24.0 * c.eps, f48d = 48.0 * c.eps, f8c2d = 8.0 * c.eps * c.c2 / c.sig2;
  const double e4d = 4.0 * c.eps, c2sd = c.c2 / c.sig2;
  const int n_own = S.own1 - S.own0;
  for (int o = grp; __any_sync(0xffffffffu, o < n_own); o += kGroups) {
    const bool valid = o < n_own;
    AccF a = {};
    double dfx = 0.0, dfy = 0.0, dfz = 0.0, dpe = 0.0, dvir = 0.0;
    int gi = 0;
    if (valid) {
      const int l = S.own0 + o;
      gi = S.gown0 + o;
      uint2 row;
      if (WHOLE) {
        row = rows[gi];
      } else {
        row = s_rows[S.row_off + o];
        row.x -= S.list_base;
        if (row.x + row.y > S.list_len) {  // inconsistent row: record and skip
          if (lane == 0) atomicOr(status, LJ_ST_LIST_OVERFLOW);
          row.y = 0;
        }
      }
      // the row's pairs; one instance per memory space of the list (in_smem: staged segment)
      auto row_pairs = [&](const uint16_t* __restrict__ el, bool in_smem) {
      if (MIXED) {
        // staged fixed-point records by 32-bit shared address: record j at a_pos + 16 j
        const uint32_t a_pos = smem_addr(sh_pos);
        const uint4 qi = lds_u4(a_pos + 16u * l);
        float4* F = (float4*)fout;
        auto pairs_at = [&](uint32_t j0, uint32_t j1, bool two) {
          pair2_q<HALF, ENERGY, WHOLE>(qi, lds_u4(a_pos + (j0 << 4)), lds_u4(a_pos + (j1 << 4)), two, c, g, a, F);
        };
        if (in_smem) {
          // list segment staged: entries by 32-bit shared address, two per iteration
          uint32_t p = smem_addr(s_ent) + 2u * (row.x + lane);
          const uint32_t pend = smem_addr(s_ent) + 2u * (row.x + row.y);
          for (; p + 2u * LANES < pend; p += 4u * LANES) pairs_at(lds_u16(p), lds_u16(p + 2u * LANES), true);
          if (p < pend) {
            const uint32_t j = lds_u16(p);
            pairs_at(j, j, false);
          }
        } else {
          unsigned e = lane;
          for (; e + LANES < row.y; e += 2 * LANES) pairs_at(el[row.x + e], el[row.x + e + LANES], true);
          if (e < row.y) pairs_at(el[row.x + e], el[row.x + e], false);
        }
      } else {
        const dvec4 qi = ((const dvec4*)sh_pos)[l];
        for (unsigned e = lane; e < row.y; e += LANES) {
          const int j = el[row.x + e];
          const dvec4 qj = ((const dvec4*)sh_pos)[j];  // its image already in place (tiles)
          double dx = qj.x - qi.x, dy = qj.y - qi.y, dz = qj.z - qi.z;
          if (WHOLE) {
            dx = fma(-rint(dx * g.inv_L64), g.L, dx);
            dy = fma(-rint(dy * g.inv_L64), g.L, dy);
            dz = fma(-rint(dz * g.inv_L64), g.L, dz);
          }
          const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
          const double ri2 = rcp_nr64(r2);
          const double si = c.sig2 * ri2;
          const double s3i = si * si * si;
          const bool in = r2 < c.rc2;
          double ff = fma(ri2 * s3i, fma(-f48d, s3i, f24d), f8c2d);
          ff = in ? ff : 0.0;
          dfx = fma(ff, dx, dfx);
          dfy = fma(ff, dy, dfy);
          dfz = fma(ff, dz, dfz);
          if (HALF) {
            dvec4* F = (dvec4*)fout;
            const int gj = sh_gid[j];
            atomicAdd(&F[gj].x, -ff * dx);
            atomicAdd(&F[gj].y, -ff * dy);
            atomicAdd(&F[gj].z, -ff * dz);
          }
          if (ENERGY) {
            const double v = e4d * fma(s3i, s3i - 1.0, fma(c2sd, r2, c.c0));
            dpe += in ? v : 0.0;
            dvir = fma(-ff, r2, dvir);
          }
        }
      }
      };
      if (WHOLE) row_pairs(ent, false);
      else if (!LONGLIST || row.x + row.y <= (unsigned)list_cap) row_pairs(s_ent, true);
      else row_pairs(ent + S.list_base, false);  // the end of a long segment stays in HBM
    }
    if (MIXED) {
      float fx = gsum<LANES>(a.fx.x + a.fx.y);
      float fy = gsum<LANES>(a.fy.x + a.fy.y);
      float fz = gsum<LANES>(a.fz.x + a.fz.y);
      if (valid && lane == 0) {
        if (HALF) atomicAdd(&((float4*)fout)[gi], make_float4(-fx, -fy, -fz, 0.0f));
        else ((float4*)fout)[gi] = make_float4(fx, fy, fz, 0.0f);
      }
      if (ENERGY) {  // the group's lanes reduce in FP32, one lane accumulates
        const float pe = c.e4 * gsum<LANES>(a.pe.x + a.pe.y), vir = -gsum<LANES>(a.vir.x + a.vir.y);
        if (lane == 0) eacc.add32(pe, vir);
      }
    } else {
      dfx = gsum<LANES>(dfx);
      dfy = gsum<LANES>(dfy);
      dfz = gsum<LANES>(dfz);
      if (valid && lane == 0) {
        dvec4* F = (dvec4*)fout;
        if (HALF) {
          atomicAdd(&F[gi].x, dfx);
          atomicAdd(&F[gi].y, dfy);
          atomicAdd(&F[gi].z, dfz);
        } else {
          F[gi] = make_dvec4(dfx, dfy, dfz, 0.0);
        }
      }
      if (ENERGY) {
        eacc.pe += dpe;
        eacc.vir += dvir;
      }
    }
  }
}

// Bookkeeping of one tile before its copies are issued: segment of the list, cell bounds,
// capacity checks (identical in every thread).  Returns whether the tile can be staged.
__device__ __forceinline__ bool force_tile_prepare(const TileInfo& ti, int64_t t, const TileArgs& ta,
                                                   const uint32_t* __restrict__ cs,
                                                   const uint2* __restrict__ tile_list, TileShared& S,
                                                   int32_t* __restrict__ status) {
  if (threadIdx.x == blockDim.x - 1) {
    const uint2 tl = tile_list[t];
    S.list_base = tl.x;
    S.list_len = tl.y;
  }
  if (!stage_offsets(ti, ta, cs, S)) {
    if (threadIdx.x == 0) atomicOr(status, LJ_ST_CELL_RANGE);
    return false;
  }
  if (S.own1 - S.own0 > ta.max_own || S.list_len > (unsigned)ta.max_list) {
    if (threadIdx.x == 0) atomicOr(status, LJ_ST_LIST_OVERFLOW);
    return false;
  }
  return true;
}

// Force over the list, tile by tile: a tile's copies overlap the arithmetic of the SM's other CTAs.
// Energies: per-thread FP64 sums -> one partial per block.
template <bool MIXED, int LANES, bool HALF, bool ENERGY, bool WHOLE, bool LONGLIST>
__global__ void __launch_bounds__(kTileThreads, 4)
    k_force_tile(const void* __restrict__ pos, const uint32_t* __restrict__ cs, int64_t N, Geom g, TileArgs ta,
                 LJConst c, const uint2* __restrict__ rows, const uint2* __restrict__ tile_list,
                 const uint16_t* __restrict__ ent, void* __restrict__ fout, double* __restrict__ part,
                 int32_t* __restrict__ status, const int* __restrict__ skip) {
  if (skip && *skip) return;  // a device-decided run stopped before this step
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ TileShared S;
  __shared__ __align__(8) uint64_t bar;
  const TileLayout L = tile_layout(ta, MIXED, true, !MIXED && (HALF || WHOLE));
  EAcc eacc;
  eacc.vscale = g.qu;
  if (WHOLE) {
    if (blockIdx.x == 0) {
      stage_whole<MIXED, !MIXED>(N, pos, S, smem, L);
      __syncthreads();
      force_tile_compute<MIXED, LANES, HALF, ENERGY, true, false>(S, smem, L, rows, ent, c, g, fout, status, eacc,
                                                                  ta.list_cap);
    }
  } else {
    if (threadIdx.x == 0) {
      mbar_init(&bar, 1);
      fence_proxy_async_smem();
    }
    __syncthreads();
    uint32_t ph = 0;
    for (int64_t t = blockIdx.x; t < ta.ntiles; t += gridDim.x) {
      const TileInfo ti = tile_info(t, ta);
      if (force_tile_prepare(ti, t, ta, cs, tile_list, S, status)) {
        stage_issue<MIXED, true>(ti, ta, pos, rows, ent, S, smem, L, &bar);
        if (!stage_finish<MIXED, true>(ti, ta, g, S, smem, L, &bar, ph, !MIXED && HALF, status)) return;
        force_tile_compute<MIXED, LANES, HALF, ENERGY, false, LONGLIST>(S, smem, L, rows, ent, c, g, fout, status, eacc,
                                                                        ta.list_cap);
      }
      __syncthreads();
    }
  }
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
// Pair work by queues.  A warp takes a run of consecutive keys.  It first filters their rows in FP32
// (differences of fixed-point copies, r_c^2 widened by what the copies' rounding, an absolute u each, and
// the FP32 arithmetic can err: filter_cut2) and queues the kept (key, partner) pairs in shared memory;
// then each lane evaluates a contiguous share of the queue, so that at most the last pair of a lane
// idles and a key's sum needs no shuffles.  A lane stores the partial sum of a key that began in an earlier
// lane in its head slot, every other one in the key's slot; the key's own lane adds slot and heads in
// lane order, so the sums do not depend on timing.  The exact r^2 < r_c^2 test is still the pair's own.
// This pays where a pair inside r_c is dear against the filter: in the FP64 form (the FP64 pipe takes 2
// lanes per clock per SM, 1/64 of the FP32 rate, whatever the number of active lanes) and in the adjoint
// pass (about 75 instructions a pair).
constexpr int kDpThreads = 128;
constexpr int kDpWarps = kDpThreads / 32;
constexpr int kDpQueue = 288;  // queued pairs per warp: nine a lane (the smallest that keeps four FP64 CTAs per SM)

template <int NACC, bool DIRECT>
struct DpWarp {
  double seg[32][NACC];       // per key: the partial sum of the lane in which its run begins
  double head[32][NACC]; // per lane: the partial sum of a run begun in an earlier lane
  uint32_t q[kDpQueue];  // key of the warp's run << 16 | staged partner
};
template <int NACC>
struct DpWarp<NACC, true> {
  uint32_t q[kDpQueue];
};

// Shared memory of an FP64 tile: FP64 positions, fixed-point records (sorted index in w), own rows,
// list segment, the warps' queues.
struct DpLayout {
  size_t xq, warp, total;
  TileLayout L;  // pos, rows, ent as the staging helpers take them
};
template <int NACC, bool DIRECT>
__host__ __device__ __forceinline__ DpLayout dp_layout(const TileArgs& ta) {
  DpLayout D;
  const size_t ms = (size_t)ta.max_staged;
  D.L.pos = 0;
  size_t o = align16(ms * 32);
  D.xq = D.L.gid = o;
  o += ms * 16;
  D.L.rows = o;
  o += align16(8 * ((size_t)ta.max_own + 2));
  D.L.ent = D.L.cnt = o;
  o += align16(2 * (size_t)ta.list_cap);
  D.warp = o;
  o += sizeof(DpWarp<NACC, DIRECT>) * kDpWarps;
  D.total = D.L.total = align16(o);
  return D;
}

// Wait (bounded, all threads) for a staged FP64 tile, put the periodic images in place and write the
// fixed-point records of the staged positions (integer operations on the FP64 bits: reading the
// records from HBM would cost 16 B per staged particle and a second array).  False on timeout.
__device__ __forceinline__ bool dp_stage_finish(const TileInfo& ti, const TileArgs& ta, const Geom& g, TileShared& S,
                                                unsigned char* smem, const DpLayout& D, uint64_t* bar, uint32_t& phase,
                                                int32_t* status) {
  bool ok = true;
  if (threadIdx.x == 0) ok = mbar_wait(bar, phase, wait_budget());
  ok = __syncthreads_and(ok) != 0;
  if (!ok) {
    if (threadIdx.x == 0) {
      atomicOr(status, LJ_ST_TIMEOUT);
      mbar_wait(bar, phase, kWaitBudget);  // let copies in flight land before the CTA leaves
    }
    __syncthreads();
    return false;
  }
  phase ^= 1u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, ncol = S.ncol;
  // a column's cells are contiguous in the sorted arrays except where z wraps: up to three runs of
  // one image each (as stage_issue copies them)
  const int cut0 = ti.z0 == 0 ? 1 : 0, cut1 = ti.z0 + ti.Tp == ta.n ? ncol - 1 : ncol;
  for (int k = warp; k < 9; k += (int)(blockDim.x >> 5)) {
    int sx, sy;
    wrap_cell(ti.cx + k / 3 - 1, ta.n, sx);
    wrap_cell(ti.cy + k % 3 - 1, ta.n, sy);
#pragma unroll 1
    for (int r = 0; r < 3; ++r) {
      const int m0 = r == 0 ? 0 : (r == 1 ? cut0 : cut1), m1 = r == 0 ? cut0 : (r == 1 ? cut1 : ncol);
      if (m1 <= m0) continue;
      const int sz = r == 0 ? -1 : (r == 2 ? 1 : 0);
      const int a = S.offq[k * ncol + m0], b = S.offq[k * ncol + m1], gq = S.g0[k * ncol + m0];
      for (int s = a + lane; s < b; s += 32) {
        dvec4* w = (dvec4*)(smem + D.L.pos) + s;
        dvec4 p = *w;
        if ((sx | sy | sz) != 0) {  // the image itself: one rounding per staged coordinate, none per pair
          if (sx != 0) p.x += sx > 0 ? g.L : -g.L;
          if (sy != 0) p.y += sy > 0 ? g.L : -g.L;
          if (sz != 0) p.z += sz > 0 ? g.L : -g.L;
          *w = p;
        }
        ((uint4*)(smem + D.xq))[s] =
            make_uint4(fixq(p.x, g.qk), fixq(p.y, g.qk), fixq(p.z, g.qk), (uint32_t)(gq + (s - a)));
      }
    }
  }
  // these generic writes precede later bulk copies into the same bytes
  fence_proxy_async_smem();
  __syncthreads();
  return true;
}

// The listed pairs of a staged tile's keys inside r_c (or within the filter's margin of it).
// sq: the staged records; W: the warp's queue.  key(o) loads what a pair needs of own key o, partner(slot)
// what it needs of the partner (a pair ahead of its use), pair(key, partner, acc) adds one pair to the key's
// NACC sums, done(o, acc) receives the sums of own key o.  ent_s: the staged part of the tile's segment, its
// first cap entries; rows beyond it are read from ent_g.
// DIRECT: done(o, acc) is called by the lanes themselves with each partial sum (it must add atomically).
template <int NACC, bool DIRECT, class Key, class Partner, class Pair, class Done>
__device__ __forceinline__ void queue_tile_pairs(const TileShared& S, const uint4* sq, const uint2* s_rows,
                                                 DpWarp<NACC, DIRECT>& W, const uint16_t* ent_s,
                                                 const uint16_t* ent_g, unsigned cap, float cut2, int32_t* status,
                                                 Key&& key, Partner&& partner, Pair&& pair, Done&& done) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  s_rows += S.row_off;
  const int n_own = S.own1 - S.own0;
  const int per = min(32, (n_own + kDpWarps - 1) / kDpWarps);  // keys per warp and turn
  for (int b0 = warp * per; b0 < n_own; b0 += kDpWarps * per) {
    const int nk = min(per, n_own - b0);
    double tot[NACC];  // lane k: the sums of key b0 + k
#pragma unroll
    for (int q = 0; q < NACC; ++q) tot[q] = 0.0;
    int ka = 0, kb = 0, cnt = 0;  // lane k: the key's range of the queue; queued pairs
    auto drain = [&]() {
      __syncwarp();
      const int c = (cnt + 31) >> 5, lo = lane * c, hi = min(lo + c, cnt);
      double acc[NACC];
      int kc = -1;
      bool head = lo > 0 && lo < cnt && (W.q[lo - 1] >> 16) == (W.q[lo] >> 16);
      auto ki = key(b0);
      auto put = [&]() {
        if constexpr (DIRECT) {
          done(b0 + kc, acc);
        } else {
          double* dst = head ? W.head[lane] : W.seg[kc];
#pragma unroll
          for (int q = 0; q < NACC; ++q) dst[q] = acc[q];
          head = false;
        }
      };
      uint32_t w = lo < hi ? W.q[lo] : 0u;
      auto pj = partner((int)(w & 0xffffu));
      for (int t = lo; t < hi; ++t) {
        const uint32_t wn = t + 1 < hi ? W.q[t + 1] : w;
        const auto pn = partner((int)(wn & 0xffffu));
        const int k = (int)(w >> 16);
        if (k != kc) {
          if (kc >= 0) put();
          kc = k;
          ki = key(b0 + k);
#pragma unroll
          for (int q = 0; q < NACC; ++q) acc[q] = 0.0;
        }
        pair(ki, pj, acc);
        w = wn;
        pj = pn;
      }
      if (kc >= 0) put();
      __syncwarp();
      if constexpr (!DIRECT) {
        if (kb > ka) {
          const int l0 = ka / c, l1 = (kb - 1) / c;
#pragma unroll
          for (int q = 0; q < NACC; ++q) tot[q] += W.seg[lane][q];
          for (int l = l0 + 1; l <= l1; ++l) {
#pragma unroll
            for (int q = 0; q < NACC; ++q) tot[q] += W.head[l][q];
          }
        }
        __syncwarp();
      }
      ka = kb = cnt = 0;
    };
    uint2 row = make_uint2(0u, 0u);
    if (lane < nk) {
      row = s_rows[b0 + lane];
      row.x -= S.list_base;
      if (row.x + row.y > S.list_len) {  // inconsistent row: record and skip
        atomicOr(status, LJ_ST_LIST_OVERFLOW);
        row.y = 0;
      }
    }
    for (int k = 0; k < nk; ++k) {
      const int start = (int)__shfl_sync(0xffffffffu, row.x, k), len = (int)__shfl_sync(0xffffffffu, row.y, k);
      const uint16_t* ent = (unsigned)(start + len) <= cap ? ent_s : ent_g;
      const uint4 qi = sq[S.own0 + b0 + k];
      if (lane == k) ka = cnt;
      for (int e0 = 0; e0 < len; e0 += 32) {
        if (cnt > kDpQueue - 32) {
          if (lane == k) kb = cnt;
          drain();
        }
        const int e = e0 + lane;
        uint32_t j = 0;
        bool in = false;
        if (e < len) {
          j = ent[start + e];
          const uint4 qj = sq[j];
          const float dx = qdiff(qj.x, qi.x), dy = qdiff(qj.y, qi.y), dz = qdiff(qj.z, qi.z);
          in = fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < cut2;
        }
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (in) W.q[cnt + __popc(m & lt)] = ((uint32_t)k << 16) | j;
        cnt += __popc(m);
      }
      if (lane == k) kb = cnt;
    }
    if (cnt > 0) drain();
    if constexpr (!DIRECT) {
      if (lane < nk) done(b0 + lane, tot);
    }
  }
}

// The same on a staged FP64 tile: pair(FP64 position of the key, partner slot, acc).
template <int NACC, bool DIRECT, class Pair, class Done>
__device__ __forceinline__ void dp_tile_pairs(const TileShared& S, const unsigned char* smem, const DpLayout& D,
                                              const uint16_t* ent_g, unsigned cap, float cut2, int32_t* status,
                                              Pair&& pair, Done&& done) {
  const dvec4* sp = (const dvec4*)(smem + D.L.pos) + S.own0;
  queue_tile_pairs<NACC, DIRECT>(
      S, (const uint4*)(smem + D.xq), (const uint2*)(smem + D.L.rows),
      ((DpWarp<NACC, DIRECT>*)(smem + D.warp))[threadIdx.x >> 5], (const uint16_t*)(smem + D.L.ent), ent_g, cap,
      cut2, status, [&](int o) { return sp[o]; }, [](int j) { return j; }, pair, done);
}

// The FP64 comparison r^2 < r_c^2 of two non-negative values by their bit patterns (the order is the
// same; a NaN compares as not inside), which takes no slot of the FP64 pipe.
__device__ __forceinline__ bool inside_rc(double r2, double rc2) {
  return __double_as_longlong(r2) < __double_as_longlong(rc2);
}

// 1/x in FP64 from the hardware approximation (rcp.approx.ftz.f64) refined by one third-order step
// r' = r + r (e + e^2), e = 1 - x r, whose error is e^3: three FP64 operations where two Newton
// steps take four.
__device__ __forceinline__ double rcp_cubic64(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// r_c^2 for the queues' filter, in units of u^2: a distance between fixed-point copies is within sqrt(3) u of the
// true one (each coordinate is rounded by at most u / 2), and its FP32 square and this figure within a relative
// 1e-6.  The absolute term counts where u is not small against r_c: lengths far below one unit (u is 2^-30 at
// least) and cells far longer than r_c.
__device__ __forceinline__ float filter_cut2(const LJConst& c) {
  const float r = sqrtf(c.rc2q) + 2.0f;
  return r * r * 1.000004f;
}

// One pair of the FP64 form's force, its sums over pairs (r^-6, r^-12, r^2 and their number, from which
// the energies come) and the scattered sums of the half list.
template <bool HALF, bool ENERGY>
struct DpForce {
  double rc2, f8c2, f24s, f48s;
  float cut2;
  double s6 = 0.0, s12 = 0.0, s2 = 0.0;
  int np = 0;
  const dvec4* sp;
  const uint4* sq;
  dvec4* fout;
  __device__ __forceinline__ DpForce(const LJConst& c, const unsigned char* smem, const DpLayout& D, dvec4* f) {
    const double sig6 = c.sig2 * c.sig2 * c.sig2;
    rc2 = c.rc2;
    f8c2 = 8.0 * c.eps * c.c2s;
    f24s = 24.0 * c.eps * sig6;
    f48s = 48.0 * c.eps * sig6 * sig6;
    cut2 = filter_cut2(c);
    sp = (const dvec4*)(smem + D.L.pos);
    sq = (const uint4*)(smem + D.xq);
    fout = f;
  }
  __device__ __forceinline__ void pair(const dvec4& qi, int j, double* acc) {
    const dvec4 qj = sp[j];
    // the half list takes d = x_i - x_j, so that ff d is the force on the partner
    const double dx = HALF ? qi.x - qj.x : qj.x - qi.x, dy = HALF ? qi.y - qj.y : qj.y - qi.y,
                 dz = HALF ? qi.z - qj.z : qj.z - qi.z;
    const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
    if (!inside_rc(r2, rc2)) return;
    const double ri2 = rcp_cubic64(r2);
    const double ri4 = ri2 * ri2, ri6 = ri4 * ri2;
    const double ff = fma(ri4 * ri4, fma(-f48s, ri6, f24s), f8c2);
    if (HALF) {
      dvec4* F = fout + sq[j].w;
      const double fx = ff * dx, fy = ff * dy, fz = ff * dz;
      acc[0] -= fx;
      acc[1] -= fy;
      acc[2] -= fz;
      atomicAdd(&F->x, fx);
      atomicAdd(&F->y, fy);
      atomicAdd(&F->z, fz);
    } else {
      acc[0] = fma(ff, dx, acc[0]);
      acc[1] = fma(ff, dy, acc[1]);
      acc[2] = fma(ff, dz, acc[2]);
    }
    if (ENERGY) {
      s6 += ri6;
      s12 = fma(ri6, ri6, s12);
      s2 += r2;
      ++np;
    }
  }
  __device__ __forceinline__ void add(int64_t i, const double* acc) const {
    dvec4* F = fout + i;
    atomicAdd(&F->x, acc[0]);
    atomicAdd(&F->y, acc[1]);
    atomicAdd(&F->z, acc[2]);
  }
};

// PE and virial from the sums over pairs: V = 4 eps (sigma^12 r^-12 - sigma^6 r^-6 + c2 r^2 / sigma^2 + c0).
__device__ __forceinline__ void dp_energies(const LJConst& c, double s6, double s12, double s2, double n, double& pe,
                                            double& vir) {
  const double sig6 = c.sig2 * c.sig2 * c.sig2, sig12 = sig6 * sig6;
  pe = 4.0 * c.eps * fma(sig12, s12, fma(-sig6, s6, fma(c.c2s, s2, c.c0 * n)));
  vir = c.eps * fma(48.0 * sig12, s12, fma(-24.0 * sig6, s6, -8.0 * c.c2s * s2));
}

// ---------------------------------------------------------------------------------------------
// Launch shapes.
static inline int sm_count() {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

static inline int tile_grid(const TileArgs& ta, int per_sm) {
  int64_t b = (int64_t)sm_count() * per_sm;
  if (b > ta.ntiles) b = ta.ntiles;
  if (b > kMaxRedBlocks) b = kMaxRedBlocks;
  return (int)(b < 1 ? 1 : b);
}

template <class K>
static void set_smem(K kernel, size_t bytes) {
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// CTAs of a kernel resident per SM at the given dynamic shared memory (registers included).
template <class K>
static int resident_per_sm(K kernel, int threads, size_t smem) {
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, threads, smem) != cudaSuccess || nb < 1) nb = 1;
  return nb;
}

static inline int per_sm_for(size_t smem_bytes) {
  int dev = 0, smem_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  int k = (int)(smem_sm / (int)(smem_bytes + sizeof(TileShared) + 1024));
  return k < 1 ? 1 : (k > 4 ? 4 : k);
}

}  // namespace ljmd
