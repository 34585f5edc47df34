// Small boxes: the whole reordering before a list construction in one cooperative launch.
#include "tile.cuh"

namespace ljmd {

// Fold, label and count, scan, scatter, rank by id, gather and position copies, tile sizes: the kernels of
// kernels_grid.cu, whose few microseconds each are launch and latency when the box is small.  A thread keeps
// its particle through all phases (its position is read once, its slot in the cell is the count's own atomic),
// every CTA scans the cell counts for itself in shared memory, and a particle goes straight to its place, the
// number of smaller ids in its cell, where the gather would have to find it.  Two grid barriers (bounded).
// The counts are zero between launches: they are cleared once every CTA has scanned them.  A
// construction as eleven launches and two host round trips took 83 us at 4,000 particles and 118 us at 32,000;
// with this kernel, the list kernel and one round trip 46 and 65 us.
constexpr int kSortThreads = 256;

__device__ __forceinline__ bool sort_barrier(GridCtl* ctl, unsigned target) {
  __syncthreads();
  bool ok = true;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&ctl->arrived, 1u);
    const long long budget = wait_budget(), t0 = clock64();
    for (;;) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&ctl->arrived) : "memory");
      if (v >= target) break;
      if (clock64() - t0 > budget) {
        atomicOr(&ctl->status, LJ_ST_TIMEOUT);
        ok = false;
        break;
      }
    }
  }
  return __syncthreads_and(ok ? 1 : 0) != 0;
}

template <bool MIXED>
__global__ void __launch_bounds__(kSortThreads) k_sort(SortArgs a) {
  __shared__ uint32_t cs[kSortCells + 1];  // counts, then cell starts
  __shared__ uint32_t sh[kSortThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t N = a.N, i = blockIdx.x * (int64_t)kSortThreads + tid;
  const Geom& g = a.g;
  GridCtl* ctl = a.ctl;
  double xs[3];
  int im[3];
  uint32_t cell = 0xffffffffu, slot = 0;
  int my_id = 0;
  if (i < N) {
    const double top = g.offset + g.L;
    int c[3];
    bool bad = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      xs[k] = a.x[k * N + i];
      im[k] = a.img[k * N + i];
    }
    my_id = a.id[i];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      bad |= !finite_d(xs[k]);
      if (cmp_ge_d(xs[k], top)) {
        xs[k] -= g.L;
        im[k] += 1;
      } else if (!cmp_ge_d(xs[k], g.offset)) {
        xs[k] += g.L;
        im[k] -= 1;
      }
      const double rel = xs[k] - g.offset;  // exact: both in [offset/2, 2 offset)
      const int ck = floor_to_int(rel * g.inv_h);
      c[k] = ck < 0 ? 0 : (ck >= g.n ? g.n - 1 : ck);
    }
    if (bad) {
      atomicOr(&ctl->status, LJ_ST_NONFINITE);
      c[0] = c[1] = c[2] = 0;
    }
    cell = ((uint32_t)c[0] * (uint32_t)g.n + (uint32_t)c[1]) * (uint32_t)g.n + (uint32_t)c[2];
  }
  {
    const unsigned peers = __match_any_sync(0xffffffffu, cell);
    const int leader = __ffs(peers) - 1;
    uint32_t base = 0;
    if (lane == leader && i < N) base = atomicAdd(&a.count[cell], (uint32_t)__popc(peers));
    slot = __shfl_sync(0xffffffffu, base, leader) + (uint32_t)__popc(peers & ((1u << lane) - 1u));
  }
  if (!sort_barrier(ctl, gridDim.x)) return;
  // exclusive scan of the counts
  for (int q = tid; q < a.ncells; q += kSortThreads) cs[q] = __ldcg(a.count + q);
  __syncthreads();
  uint32_t mx = 0;
  {
    const int per = (a.ncells + kSortThreads - 1) / kSortThreads, q0 = min(tid * per, a.ncells), q1 = min(q0 + per, a.ncells);
    uint32_t t = 0;
    for (int q = q0; q < q1; ++q) {
      t += cs[q];
      mx = max(mx, cs[q]);
    }
    uint32_t inc = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) sh[warp] = inc;
    __syncthreads();
    uint32_t run = inc - t;
    for (int w = 0; w < warp; ++w) run += sh[w];
    for (int q = q0; q < q1; ++q) {
      const uint32_t m = cs[q];
      cs[q] = run;
      run += m;
    }
    if (tid == kSortThreads - 1) cs[a.ncells] = run;
  }
  __syncthreads();
  if (i < N) a.cell_ids[cs[cell] + slot] = my_id;
  if (!sort_barrier(ctl, 2 * gridDim.x)) return;
  // the particle's place and its state there
  if (i < N) {
    const uint32_t b = cs[cell], e = cs[cell + 1];
    uint32_t p = b;
    for (uint32_t q = b; q < e; ++q) p += __ldcg(a.cell_ids + q) < my_id ? 1u : 0u;
    float4 h;
    float unused;
    split_hi_lo(xs[0], h.x, unused);
    split_hi_lo(xs[1], h.y, unused);
    split_hi_lo(xs[2], h.z, unused);
    h.w = __int_as_float((int)p);
    a.hi[p] = h;
    if constexpr (MIXED) {
      const uint4 r = make_uint4(fixq(xs[0], g.qk), fixq(xs[1], g.qk), fixq(xs[2], g.qk), p);
      ((uint4*)a.pos)[p] = r;
      ((uint4*)a.ref)[p] = r;
      ((float4*)a.f2)[p] = ((const float4*)a.f)[i];
    } else {
      const dvec4 r = make_dvec4(xs[0], xs[1], xs[2], 0.0);
      ((dvec4*)a.pos)[p] = r;
      ((dvec4*)a.ref)[p] = r;
      ((dvec4*)a.f2)[p] = ((const dvec4*)a.f)[i];
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      a.x2[k * N + p] = xs[k];
      a.v2[k * N + p] = a.v[k * N + i];
      a.img2[k * N + p] = im[k];
    }
    a.id2[p] = my_id;
  }
  const int64_t threads = (int64_t)gridDim.x * kSortThreads;
  for (int64_t q = i; q < a.ncells; q += threads) {
    a.cell_start[q] = cs[q];
    a.cell_count[q] = cs[q + 1] - cs[q];
    a.count[q] = 0u;
  }
  if (i == 0) a.cell_start[a.ncells] = cs[a.ncells];
  // tile sizes (as k_tile_sizes); the last CTA compares them with the capacities of the waiting list kernel
  unsigned mst = 0, mown = 0;
  for (int64_t t = i; t < a.ta.ntiles; t += threads) {
    const TileInfo ti = tile_info(t, a.ta);
    const int ncol = ti.Tp + 2;
    unsigned tot = 0;
    for (int q = 0; q < 9 * ncol; ++q) {
      int sx, sy, sz;
      const uint32_t c = cell_of_q(ti, a.ta.n, ncol, q, sx, sy, sz);
      tot += cs[c + 1] - cs[c];
    }
    const uint32_t c0 = ((uint32_t)ti.cx * (uint32_t)a.ta.n + (uint32_t)ti.cy) * (uint32_t)a.ta.n + (uint32_t)ti.z0;
    mst = max(mst, tot);
    mown = max(mown, cs[c0 + ti.Tp] - cs[c0]);
  }
  mst = __reduce_max_sync(0xffffffffu, mst);
  mown = __reduce_max_sync(0xffffffffu, mown);
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) {
    if (mst) atomicMax(&ctl->sizes[0], mst);
    if (mown) atomicMax(&ctl->sizes[1], mown);
    if (blockIdx.x == 0) atomicMax(&ctl->sizes[2], mx);
    __threadfence();
  }
  __syncthreads();
  if (tid == 0 && atomicAdd(&ctl->ticket, 1u) == gridDim.x - 1) {
    __threadfence();
    const unsigned staged = atomicMax(&ctl->sizes[0], 0u), own = atomicMax(&ctl->sizes[1], 0u), mc = atomicMax(&ctl->sizes[2], 0u);
    ctl->ok = a.caps && staged <= (unsigned)a.ta.max_staged && own <= (unsigned)a.ta.max_own &&
              9u * ((3u * mc + 31u) / 32u) + 1u <= (unsigned)a.ta.max_chunks;
  }
}

// Particles that one launch takes (its grid has to be resident), 0 if it cannot run.
int64_t sort_capacity() {
  static int64_t cap = -1;
  if (cap < 0) {
    int dev = 0, coop = 0, a = 0, b = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (!coop || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_sort<true>, kSortThreads, 0) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_sort<false>, kSortThreads, 0) != cudaSuccess) {
      cudaGetLastError();
      a = b = 0;
    }
    cap = (int64_t)std::min(a, b) * sm_count() * kSortThreads;
  }
  return cap;
}

int64_t sort_grid(int64_t N) { return (N + kSortThreads - 1) / kSortThreads; }

// 0: launched; 1: the device cannot hold the grid now (nothing done); -1: error.
int launch_sort(int precision, SortArgs a, cudaStream_t s) {
  const unsigned grid = (unsigned)sort_grid(a.N);
  void* args[] = {&a};
  const cudaError_t e =
      cudaLaunchCooperativeKernel(precision == LJ_MIXED ? (const void*)k_sort<true> : (const void*)k_sort<false>,
                                  dim3(grid), dim3(kSortThreads), args, 0, s);
  return e == cudaSuccess ? 0 : (e == cudaErrorCooperativeLaunchTooLarge ? 1 : -1);
}

int set_wait_budget_sort(long long cycles) { return set_unit_wait_budget(cycles); }

}  // namespace ljmd
