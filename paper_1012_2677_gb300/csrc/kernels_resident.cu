// Resident runs: velocity-Verlet steps of a box whose tiles all fit on the chip at once, as one
// cooperative launch.  Each CTA keeps one tile: its particles' positions, velocities and forces, its rows
// and its list segment stay in shared memory for the whole run.  A step is
//   kick and drift of the tile's own particles (FP64), their position copies written to global memory
//     (two buffers, taken in turn) and the largest displacement reduced;
//   a grid barrier;
//   the list-validity rule (every CTA reads the same maximum and decides the same); the copies of the
//     tile's neighbour cells staged from L2, the periodic images put in place;
//   the forces of the own particles over the list.
// One barrier a step suffices: the next drift writes the other buffer, and the one after that comes
// after a barrier that every CTA reaches only when it has read this one.  The half list needs a second
// barrier, between its scattered sums and their use.  The run ends after K steps or at the drift that
// expired the list; the state, forces and energies are then what the launches of one step each leave.
//
// What bounds a small box is latency: two launches a step, each staging list, rows and bookkeeping anew
// and ending in a last-CTA reduction, took 28 us (mixed form) where the pair arithmetic is about 1 us.
// Here a step costs the barrier, one L2 read of the neighbour cells and the pair chain; the energy sums are
// taken by warps that would wait for the barrier.  100 steps of 4,000 particles with their 8 list
// constructions: mixed form 3.50 -> 1.65 ms, FP64 form 5.09 -> 3.15 ms; 50 steps of 32,003 particles
// 2.60 -> 1.47 ms.
#include "tile.cuh"

namespace ljmd {

constexpr int kResThreads = 256;  // mixed form: 3 CTAs per SM
constexpr int kResKeys = 8;       // keys per lane group, at most (FP32 energy partials are summed in FP64)

// Shared memory of a resident tile.
struct ResLayout {
  TileLayout L;         // pos (mixed: records; FP64: dvec4), rows, ent
  DpLayout D;           // FP64: records and queues for dp_tile_pairs
  size_t src;           // uint32 [max_staged]: sorted index, image code (x, y, z in two bits each) above
  size_t xv;            // double [6][max_own]
  size_t ref, f;        // uint4/dvec4 and float4/dvec4 [max_own]
  size_t ke;            // float/double [max_own]
  size_t en;            // mixed: float [2][threads]; FP64: double [3][threads], int [threads]
  size_t total;
};
template <bool MIXED, bool HALF>
__host__ __device__ __forceinline__ ResLayout res_layout(const TileArgs& ta) {
  ResLayout R;
  const size_t ms = (size_t)ta.max_staged, mo = (size_t)ta.max_own;
  size_t o;
  if (MIXED) {
    R.L.pos = 0;
    o = ms * 16;
    R.L.gid = 0;
    R.L.rows = o;
    o += align16(8 * (mo + 2));
    R.L.ent = R.L.cnt = o;
    o += align16(2 * (size_t)ta.list_cap);
    R.L.total = o;
    R.D = DpLayout{};
  } else {
    R.D = dp_layout<3, HALF>(ta);
    R.L = R.D.L;
    o = R.D.total;
  }
  R.src = o;
  o += align16(4 * ms);
  R.xv = o;
  o += align16(48 * mo);
  R.ref = o;
  o += (MIXED ? 16 : 32) * mo;
  R.f = o;
  o += (MIXED ? 16 : 32) * mo;
  R.ke = o;
  o += align16((MIXED ? 4 : 8) * mo);
  R.en = o;
  o += MIXED ? 8 * kResThreads : 28 * kDpThreads;
  R.total = align16(o);
  return R;
}

constexpr int kImageShift = 26;  // sorted indices below 2^26 (a resident box is far smaller)

// Image code of a staged cell: (shift + 1) per axis, two bits each.
__device__ __forceinline__ uint32_t image_code(int sx, int sy, int sz) {
  return (uint32_t)((sx + 1) | (sy + 1) << 2 | (sz + 1) << 4) << kImageShift;
}

// Grid barrier `phase` (0, 1, ...) of the run: thread 0 arrives and waits, with a bounded wait; a
// timeout marks the run so that the other CTAs leave too.
__device__ __forceinline__ bool grid_wait(ResidentCtl* ctl, unsigned phase, int32_t* status) {
  __threadfence();
  atomicAdd(&ctl->arrived, 1u);
  const unsigned target = (phase + 1u) * gridDim.x;
  const long long budget = wait_budget(), t0 = clock64();
  for (;;) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&ctl->arrived) : "memory");
    if (v >= target) return true;
    if (*(volatile int*)&ctl->abort) return false;
    if (clock64() - t0 > budget) {
      atomicOr(status, LJ_ST_TIMEOUT);
      *(volatile int*)&ctl->abort = 1;
      return false;
    }
  }
}

template <bool MIXED>
struct ResTypes;
template <>
struct ResTypes<true> {
  typedef float4 F;
  typedef uint4 P;
  typedef float E;
};
template <>
struct ResTypes<false> {
  typedef dvec4 F;
  typedef dvec4 P;
  typedef double E;
};

template <bool MIXED, bool HALF, int LANES>
__global__ void __launch_bounds__(MIXED ? kResThreads : kDpThreads, MIXED ? 3 : 4) k_resident(ResidentArgs a) {
  constexpr int NT = MIXED ? kResThreads : kDpThreads;
  typedef typename ResTypes<MIXED>::F FT;
  typedef typename ResTypes<MIXED>::P PT;
  typedef typename ResTypes<MIXED>::E ET;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ TileShared S;
  __shared__ float s_d2[NT / 32], s_v2[NT / 32];
  __shared__ int s_expired;
  __shared__ double sh[32];
  const TileArgs& ta = a.ta;
  const Geom& g = a.g;
  const ResLayout R = res_layout<MIXED, HALF>(ta);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t N = a.N;
  const int64_t rec_base = a.log ? *a.count : 0;  // before the first barrier: CTA 0 advances it at the end
  double* xv = (double*)(smem + R.xv);
  FT* s_f = (FT*)(smem + R.f);
  ET* s_ke = (ET*)(smem + R.ke);
  const TileInfo ti = tile_info(blockIdx.x, ta);
  // ---- bookkeeping, list and state of the tile
  bool ok = force_tile_prepare(ti, blockIdx.x, ta, a.cs, a.tile_list, S, a.status);
  const int n_own = ok ? S.own1 - S.own0 : 0, total = ok ? S.total : 0;
  const int mo = ta.max_own;
  if (ok) {
    uint32_t* src = (uint32_t*)(smem + R.src);
    for (int q = warp; q < S.ncell; q += NT / 32) {
      int sx, sy, sz;
      cell_of_q(ti, ta.n, S.ncol, q, sx, sy, sz);
      const uint32_t code = image_code(sx, sy, sz);
      for (int s = S.offq[q] + lane; s < S.offq[q + 1]; s += 32) src[s] = (uint32_t)(S.g0[q] + (s - S.offq[q])) | code;
    }
    const uint4* e = (const uint4*)(a.ent + S.list_base);  // segments are padded to 8 entries (16 bytes)
    for (unsigned w = tid; w < min(S.list_len, (unsigned)ta.list_cap) / 8u; w += NT) ((uint4*)(smem + R.L.ent))[w] = e[w];
  }
  if (tid == 0) {
    S.row_off = 0;
    if (!ok) *(volatile int*)&a.ctl->abort = 1;  // (recorded in the status word) the others leave too
  }
  for (int o = tid; o < n_own; o += NT) {
    const int64_t i = S.gown0 + o;
    ((uint2*)(smem + R.L.rows))[o] = a.rows[i];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      xv[k * mo + o] = a.x[k * N + i];
      xv[(3 + k) * mo + o] = a.v[k * N + i];
    }
    ((PT*)(smem + R.ref))[o] = ((const PT*)a.ref)[i];
    s_f[o] = ((const FT*)a.f)[i];
    if (HALF) ((FT*)a.f)[i] = FT{};  // the scattered sums start at zero
  }
  __syncthreads();
  const double h = 0.5 * a.dt;
  double dutc = a.ctl->dutc;  // thread 0's copy is the one used
  unsigned phase = 0;
  bool bad = false, aborted = !ok, stopped = false;
  int done = 0;
  float last_d2 = 0.0f, last_v2 = 0.0f;
  auto want = [&](int64_t t) { return a.ee > 0 && t % a.ee == 0; };
  // Kick by kpre (the full-step velocity, whose kinetic energy is taken if ke), kpost, drift by dt.
  auto integrate = [&](double kpre, double kpost, double dt, bool ke, void* pos, double* cap, float& d2max, float& v2max) {
    const double kk = kpre + kpost;
    const float kpre_f = (float)kpre;
    for (int o = tid; o < n_own; o += NT) {
      const int64_t i = S.gown0 + o;
      const FT f = s_f[o];
      const double F[3] = {MIXED ? f32_to_f64((float)f.x) : (double)f.x, MIXED ? f32_to_f64((float)f.y) : (double)f.y,
                           MIXED ? f32_to_f64((float)f.z) : (double)f.z};
      const float Ff[3] = {(float)f.x, (float)f.y, (float)f.z};
      double xs[3], ked = 0.0;
      float kef = 0.0f, vd2 = 0.0f;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        double vk = xv[(3 + k) * mo + o];
        if (ke) {
          if (MIXED) {
            const float vf = fmaf(kpre_f, Ff[k], f64_to_f32(vk));
            kef = fmaf(vf, vf, kef);
          } else {
            const double vf = fma(kpre, F[k], vk);
            ked = fma(vf, vf, ked);
          }
        }
        if (!is_zero_d(kk)) vk = fma(kk, F[k], vk);
        if (a.dutc_rule) {
          const float vs = MIXED ? f64_to_f32(vk) : (float)vk;
          vd2 = fmaf(vs, vs, vd2);
        }
        double xk = xv[k * mo + o];
        if (!is_zero_d(dt)) xk = fma(dt, vk, xk);
        xv[(3 + k) * mo + o] = vk;
        xv[k * mo + o] = xk;
        xs[k] = xk;
        bad |= !finite_d(xk) || !finite_d(vk);
      }
      if (ke) s_ke[o] = MIXED ? (ET)(0.5f * kef) : (ET)(0.5 * ked);
      if (pos) {
        v2max = fmaxf(v2max, vd2);
        const PT r = ((const PT*)(smem + R.ref))[o];
        if constexpr (MIXED) {
          const uint4 q = make_uint4(fixq(xs[0], g.qk), fixq(xs[1], g.qk), fixq(xs[2], g.qk), (uint32_t)i);
          ((uint4*)pos)[i] = q;
          const float dx = qdiff(q.x, r.x) * g.qu, dy = qdiff(q.y, r.y) * g.qu, dz = qdiff(q.z, r.z) * g.qu;
          d2max = fmaxf(d2max, fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
        } else {
          ((dvec4*)pos)[i] = make_dvec4(xs[0], xs[1], xs[2], 0.0);
          const double dx = xs[0] - r.x, dy = xs[1] - r.y, dz = xs[2] - r.z;
          d2max = fmaxf(d2max, __double2float_ru(fma(dx, dx, fma(dy, dy, dz * dz))));
        }
        if (cap) {  // the unwrapped positions of this state, id order
          const int64_t p = a.id[i];
#pragma unroll
          for (int k = 0; k < 3; ++k) cap[3 * p + k] = (xs[k] - g.offset) + (double)a.img[k * N + i] * g.L;
        }
      }
    }
  };
  // Energy partials of the tile, state of record slot k (warps 1 and 2, while warp 0 waits for the grid).
  const int groups = NT / LANES;
  auto record = [&](int k, bool pe) {
    double* out = a.rec + 3 * ((size_t)k * gridDim.x + blockIdx.x);
    if (warp == 2) {
      double s = 0.0;
      for (int o = lane; o < n_own; o += 32) s += MIXED ? f32_to_f64((float)s_ke[o]) : (double)s_ke[o];
      s = warp_sum(s);
      if (lane == 0) out[2] = s;
    } else if (warp == 1 && pe) {
      double e = 0.0, w = 0.0;
      if constexpr (MIXED) {
        const float* en = (const float*)(smem + R.en);
        for (int q = lane; q < groups; q += 32) {
          e += f32_to_f64(en[q]);
          w += f32_to_f64(en[NT + q]);
        }
        e = warp_sum(e);
        w = warp_sum(w);
      } else {
        const double* en = (const double*)(smem + R.en);
        const int* np = (const int*)(en + 3 * NT);
        double s6 = 0.0, s12 = 0.0, s2 = 0.0;
        int n = 0;
        for (int q = lane; q < NT; q += 32) {
          s6 += en[q];
          s12 += en[NT + q];
          s2 += en[2 * NT + q];
          n += np[q];
        }
        s6 = warp_sum(s6);
        s12 = warp_sum(s12);
        s2 = warp_sum(s2);
        n = __reduce_add_sync(0xffffffffu, n);
        dp_energies(a.c, s6, s12, s2, (double)n, e, w);
      }
      if (lane == 0) {
        out[0] = e;
        out[1] = w;
      }
    }
  };
  // The position copies of the tile's neighbour cells (written by other CTAs of this launch: read past L1).
  auto stage = [&](const void* P) {
    const uint32_t* src = (const uint32_t*)(smem + R.src);
#pragma unroll 4
    for (int s = tid; s < total; s += NT) {
      const uint32_t w = src[s], i = w & ((1u << kImageShift) - 1u);
      const int sx = (int)(w >> kImageShift & 3u) - 1, sy = (int)(w >> (kImageShift + 2) & 3u) - 1,
                sz = (int)(w >> (kImageShift + 4)) - 1;
      if constexpr (MIXED) {
        uint4 q = __ldcg((const uint4*)P + i);
        q.x = shift_q(q.x, sx, g);
        q.y = shift_q(q.y, sy, g);
        q.z = shift_q(q.z, sz, g);
        ((uint4*)(smem + R.L.pos))[s] = q;
      } else {
        const double2* p2 = (const double2*)((const dvec4*)P + i);
        const double2 u = __ldcg(p2), t = __ldcg(p2 + 1);
        dvec4 p = make_dvec4(u.x, u.y, t.x, 0.0);
        if (sx != 0) p.x += sx > 0 ? g.L : -g.L;
        if (sy != 0) p.y += sy > 0 ? g.L : -g.L;
        if (sz != 0) p.z += sz > 0 ? g.L : -g.L;
        ((dvec4*)(smem + R.L.pos))[s] = p;
        ((uint4*)(smem + R.D.xq))[s] = make_uint4(fixq(p.x, g.qk), fixq(p.y, g.qk), fixq(p.z, g.qk), i);
      }
    }
  };
  // Wait of all CTAs for one another; false (all threads) if the run was given up.
  auto grid_sync = [&]() {
    bool good = true;
    __syncthreads();
    if (tid == 0) good = grid_wait(a.ctl, phase, a.status);
    ++phase;
    return __syncthreads_and(good) != 0;
  };
  // Forces of the own particles from the staged tile into s_f (the half list by way of the global sums).
  auto pair_work = [&](auto energy) {
    constexpr bool E = decltype(energy)::value;
    if constexpr (MIXED) {
      float4* fout = HALF ? (float4*)a.f : (float4*)s_f - S.gown0;
      EAcc eacc;
      eacc.vscale = g.qu;
      force_tile_compute<true, LANES, HALF, E, false, true, NT>(S, smem, R.L, a.rows, a.ent, a.c, g, fout, a.status, eacc,
                                                                ta.list_cap);
      if (E && (tid & (LANES - 1)) == 0) {  // at most kResKeys keys a group: nothing folded into FP64 yet
        float* en = (float*)(smem + R.en);
        en[tid / LANES] = eacc.pe32;
        en[NT + tid / LANES] = eacc.vir32 * g.qu;
      }
    } else {
      DpForce<HALF, E> body(a.c, smem, R.D, (dvec4*)a.f);
      dp_tile_pairs<3, HALF>(
          S, smem, R.D, a.ent + S.list_base, (unsigned)ta.list_cap, body.cut2, a.status,
          [&](const dvec4& qi, int j, double* acc) { body.pair(qi, j, acc); },
          [&](int o, const double* acc) {
            if (HALF) body.add(S.gown0 + o, acc);
            else ((dvec4*)s_f)[o] = make_dvec4(acc[0], acc[1], acc[2], 0.0);
          });
      if (E) {
        double* en = (double*)(smem + R.en);
        en[tid] = body.s6;
        en[NT + tid] = body.s12;
        en[2 * NT + tid] = body.s2;
        ((int*)(en + 3 * NT))[tid] = body.np;
      }
    }
  };
  auto forces = [&](bool e_now) {
    if (e_now) pair_work(std::true_type());
    else pair_work(std::false_type());
    if (HALF) {
      if (!grid_sync()) return false;
      for (int o = tid; o < n_own; o += NT) {
        FT* p = (FT*)a.f + S.gown0 + o;
        if constexpr (MIXED) {
          s_f[o] = __ldcg(p);
        } else {
          const double2* p2 = (const double2*)p;
          const double2 u = __ldcg(p2), t = __ldcg(p2 + 1);
          s_f[o] = make_dvec4(u.x, u.y, t.x, 0.0);
        }
        *p = FT{};  // for the next step's sums, which come after the next barrier
      }
    }
    __syncthreads();
    return true;
  };
  // ---- the force of the first state, if it is not current
  if (a.need_force) {
    if (HALF && !grid_sync()) aborted = true;  // every tile's sums are zero
    if (!aborted) {
      stage(a.pos);
      __syncthreads();
      if (!forces(want(a.step0))) aborted = true;
    }
  }
  // ---- the steps
  for (int k = 0; k < a.K && !aborted; ++k) {
    void* P = (k & 1) ? a.pos : a.pos_alt;
    const bool rec = k == 0 ? a.rec0 != 0 : want(a.step0 + k);
    float d2 = 0.0f, v2 = 0.0f;
    integrate((a.first && k == 0) ? 0.0 : h, h, a.dt, rec, P,
              a.cap_x ? a.cap_x + 3 * N * (a.step0 + k + 1 - a.cap_step0) : nullptr, d2, v2);
    d2 = warp_max(d2);
    if (a.dutc_rule) v2 = warp_max(v2);
    if (lane == 0) {
      s_d2[warp] = d2;
      s_v2[warp] = v2;
    }
    __syncthreads();
    bool good = true;
    if (tid == 0) {
      for (int w = 1; w < NT / 32; ++w) {
        d2 = fmaxf(d2, s_d2[w]);
        v2 = fmaxf(v2, s_v2[w]);
      }
      atomicMax(&a.ctl->dmax[k][0], __float_as_uint(d2));
      if (a.dutc_rule) atomicMax(&a.ctl->dmax[k][1], __float_as_uint(v2));
      good = grid_wait(a.ctl, phase, a.status);
    }
    if (rec) record(k, k > 0 || a.need_force);
    ++phase;
    if (!__syncthreads_and(good)) {
      aborted = true;
      break;
    }
    if (tid == 0) {  // the validity rule, on the same values in every CTA
      last_d2 = __uint_as_float(__ldcg(&a.ctl->dmax[k][0]));
      bool expired;
      if (a.dutc_rule) {
        last_v2 = __uint_as_float(__ldcg(&a.ctl->dmax[k][1]));
        dutc -= a.two_dt * sqrt((double)last_v2) * (1.0 + 1e-6);
        expired = !(dutc > 0.0);
      } else {
        expired = last_d2 > a.limit2_lo && sqrt((double)last_d2) > a.disp_limit;
      }
      s_expired = expired;
    }
    stage(P);
    __syncthreads();
    done = k + 1;
    if (s_expired) {
      stopped = true;
      break;
    }
    if (!forces(want(a.step0 + k + 1))) aborted = true;
  }
  // ---- the end of the run
  const bool final_kick = a.last && !stopped && !aborted;
  const bool rec_last = final_kick && want(a.step0 + a.K);
  if (final_kick) {
    float d2 = 0.0f, v2 = 0.0f;
    integrate(h, 0.0, 0.0, rec_last, nullptr, nullptr, d2, v2);
    __syncthreads();
    if (rec_last) record(a.K, true);
  } else if (!stopped && !aborted && want(a.step0 + a.K)) {
    record(a.K, true);
  }
  if (!stopped && !aborted && want(a.step0 + a.K) && warp == 1 && lane == 0) {  // PE partials of the last state
    const double* out = a.rec + 3 * ((size_t)a.K * gridDim.x + blockIdx.x);
    a.part_out[2 * (size_t)blockIdx.x] = out[0];  // written by this thread
    a.part_out[2 * (size_t)blockIdx.x + 1] = out[1];
  }
  for (int o = tid; o < n_own; o += NT) {
    const int64_t i = S.gown0 + o;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      a.x[k * N + i] = xv[k * mo + o];
      a.v[k * N + i] = xv[(3 + k) * mo + o];
    }
    ((FT*)a.f)[i] = s_f[o];
    if (a.K & 1 && !stopped) ((PT*)a.pos)[i] = ((const PT*)a.pos_alt)[i];  // written by this thread
  }
  if (bad) atomicOr(a.status, LJ_ST_NONFINITE);
  if (blockIdx.x == 0 && tid == 0) {
    a.ctl->stop = stopped;
    a.ctl->stop_at = done - 1;
    a.ctl->last[0] = last_d2;
    a.ctl->last[1] = last_v2;
    a.ctl->dutc = dutc;
  }
  if (a.ee <= 0) return;
  // ---- the energy records: one CTA a record, partials summed in tile order
  __syncthreads();
  bool good = !aborted;
  if (tid == 0 && good) good = grid_wait(a.ctl, phase, a.status);
  if (!__syncthreads_and(good)) return;
  const int kmax = rec_last ? a.K + 1 : (stopped ? done : a.K);  // record slots taken: k < kmax
  auto slot = [&](int k) { return k == 0 ? a.rec0 != 0 : want(a.step0 + k); };
  int k_last = kmax - 1;
  while (k_last >= 0 && !slot(k_last)) --k_last;
  int64_t ord = rec_base;
  int r = 0;
  for (int k = 0; k <= k_last; ++k) {
    if (!slot(k)) continue;
    if (r++ % (int)gridDim.x == (int)blockIdx.x) {
      const double* q = a.rec + 3 * (size_t)k * gridDim.x;
      const bool own_pe = k > 0 || a.need_force;  // else the first state's force came from an earlier launch
      double pe = 0.0, vir = 0.0, ke = 0.0;
      for (int b = tid; b < (int)gridDim.x; b += NT) {
        if (own_pe) {
          pe += __ldcg(q + 3 * b);
          vir += __ldcg(q + 3 * b + 1);
        }
        ke += __ldcg(q + 3 * b + 2);
      }
      if (!own_pe) {
        for (int b = tid; b < a.nbf; b += NT) {
          pe += __ldcg(a.part_in + 2 * b);
          vir += __ldcg(a.part_in + 2 * b + 1);
        }
      }
      pe = block_sum(pe, sh);
      __syncthreads();
      vir = block_sum(vir, sh);
      __syncthreads();
      ke = block_sum(ke, sh);
      __syncthreads();
      if (tid == 0) {
        pe *= a.pe_scale;
        vir *= a.pe_scale;
        const double step = (double)(a.step0 + k);
        if (a.log && ord < a.log_cap) {
          a.log[4 * ord + 0] = step;
          a.log[4 * ord + 1] = pe;
          a.log[4 * ord + 2] = ke;
          a.log[4 * ord + 3] = vir;
        }
        if (k == k_last) {  // the current energies
          a.energies[0] = pe;
          a.energies[1] = ke;
          a.energies[2] = vir;
          a.energies[3] = step;
        }
      }
    }
    ++ord;
  }
  if (blockIdx.x == 0 && tid == 0 && a.log) *a.count = ord;
}

// Shape of a resident run: the threads per key, or 0 if the tiles do not all fit on the chip at once.
// Tiles of many keys leave a group of four threads eight keys at most.
template <bool MIXED, bool HALF, int LANES>
static bool resident_fits(const TileArgs& ta) {
  const size_t sm = res_layout<MIXED, HALF>(ta).total;
  int dev = 0, smem_max = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (sm + kStaticSmem > (size_t)smem_max) return false;
  set_smem(k_resident<MIXED, HALF, LANES>, sm);
  return ta.ntiles <=
         (int64_t)sm_count() * resident_per_sm(k_resident<MIXED, HALF, LANES>, MIXED ? kResThreads : kDpThreads, sm);
}
template <bool HALF>
static int resident_lanes_mixed(const TileArgs& ta) {
  if (ta.max_own <= kResThreads / 16) return resident_fits<true, HALF, 16>(ta) ? 16 : 0;
  if (ta.max_own <= kResThreads / 8) return resident_fits<true, HALF, 8>(ta) ? 8 : 0;
  if (ta.max_own <= kResKeys * kResThreads / 4) return resident_fits<true, HALF, 4>(ta) ? 4 : 0;
  return 0;
}
int resident_lanes(int precision, int half, const TileArgs& ta, int64_t N) {
  if (ta.whole || N >= (int64_t)1 << kImageShift || ta.ntiles > kMaxRedBlocks) return 0;
  if (precision == LJ_MIXED) return half ? resident_lanes_mixed<true>(ta) : resident_lanes_mixed<false>(ta);
  if (!dp_fits(ta)) return 0;
  return (half ? resident_fits<false, true, 1>(ta) : resident_fits<false, false, 1>(ta)) ? 1 : 0;
}

template <bool MIXED, bool HALF, int LANES>
static cudaError_t resident_launch(ResidentArgs& a, cudaStream_t s) {
  const size_t sm = res_layout<MIXED, HALF>(a.ta).total;
  set_smem(k_resident<MIXED, HALF, LANES>, sm);
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel((const void*)k_resident<MIXED, HALF, LANES>, dim3((unsigned)a.ta.ntiles),
                                     dim3(MIXED ? kResThreads : kDpThreads), args, sm, s);
}
template <bool HALF>
static cudaError_t resident_launch_mixed(int lanes, ResidentArgs& a, cudaStream_t s) {
  if (lanes == 16) return resident_launch<true, HALF, 16>(a, s);
  if (lanes == 8) return resident_launch<true, HALF, 8>(a, s);
  return resident_launch<true, HALF, 4>(a, s);
}
int launch_resident(int precision, int half, int lanes, ResidentArgs a, cudaStream_t s) {
  cudaError_t e;
  if (precision == LJ_MIXED) e = half ? resident_launch_mixed<true>(lanes, a, s) : resident_launch_mixed<false>(lanes, a, s);
  else e = half ? resident_launch<false, true, 1>(a, s) : resident_launch<false, false, 1>(a, s);
  return e == cudaSuccess ? 0 : (e == cudaErrorCooperativeLaunchTooLarge ? 1 : -1);
}
int set_wait_budget_resident(long long cycles) { return set_unit_wait_budget(cycles); }

}  // namespace ljmd
