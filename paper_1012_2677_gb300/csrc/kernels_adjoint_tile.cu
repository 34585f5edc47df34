// The adjoint pass over the list: Hessian-vector product, forces and parameter derivatives.
#include "tile.cuh"

namespace ljmd {

// ---------------------------------------------------------------------------------------------
// Adjoint pass over the list (the derivatives the reverse-time recurrences need), for the pair
// energy u(s) of Eq. 2 as a function of s = r^2 (a = sigma^2 / s):
//   u   = 4 eps (a^6 - a^3 + c2 s / sigma^2 + c0)
//   u'  = du/ds   = 4 eps ((3 a^3 - 6 a^6) / s + c2 / sigma^2)
//   u'' = d2u/ds2 = 4 eps (42 a^6 - 12 a^3) / s^2
//   du/dsigma  = (4 eps / sigma) (12 a^6 - 6 a^3 - 2 c2 s / sigma^2)
//   du'/dsigma = (4 eps / sigma) ((18 a^3 - 72 a^6) / s - 2 c2 / sigma^2)
// (c2, c0 fixed: r_c scales with sigma).  Per key i, with d = x_j - x_i and dw = w_i - w_j:
//   (H w)_i += 2 u' dw + 4 u'' d (d . dw)        (Hessian of the potential energy times w)
//   F_i     += 2 u' d                              (force, = -dPE/dx_i)
//   w . dF/dsigma += w_i . (2 du'/dsigma d),  w . dF/deps += w_i . (2 u' d) / eps
//   PE += u / 2,  dPE/deps += u / (2 eps),  dPE/dsigma += (du/dsigma) / 2   (full list: each pair twice)
// all zero for s >= r_c^2.  Block partials: [w.dF/deps, w.dF/dsigma, dPE/deps, dPE/dsigma, PE].
constexpr int kAdjLanes = 4;
constexpr int kAdjParts = 5;

// One key's results: H w and F to their arrays, or at once into the position adjoint (id order).
__device__ __forceinline__ void adjoint_row(const AdjointOut& out, int64_t gi, double hx, double hy, double hz, double fx,
                                            double fy, double fz) {
  if (out.lx) {
    double* l = out.lx + 3 * (int64_t)out.id[gi];
    double dx = out.c * hx, dy = out.c * hy, dz = out.c * hz;
    if (out.a != 0.0) {
      dx = fma(out.a, fx, dx);
      dy = fma(out.a, fy, dy);
      dz = fma(out.a, fz, dz);
    }
    l[0] -= dx;
    l[1] -= dy;
    l[2] -= dz;
    return;
  }
  ((dvec4*)out.hw)[gi] = make_dvec4(hx, hy, hz, 0.0);
  if (out.fo) ((dvec4*)out.fo)[gi] = make_dvec4(fx, fy, fz, 0.0);
}

// The block partials, and by the last CTA to finish their sums in block order (and their share of the
// parameter gradient, if one is being summed).
__device__ __forceinline__ void adjoint_finish(const double* acc, const AdjointOut& out, double* __restrict__ part,
                                               unsigned int* __restrict__ ticket, double* __restrict__ sums) {
  __shared__ double sh[kAdjParts][32];
  __shared__ int s_last;
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = (int)(blockDim.x >> 5);
  auto reduce = [&](double* v) {  // sums of the block in thread 0 (warp butterflies, then warp 0)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
      for (int k = 0; k < kAdjParts; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    }
    __syncthreads();
    if (l == 0) {
#pragma unroll
      for (int k = 0; k < kAdjParts; ++k) sh[k][w] = v[k];
    }
    __syncthreads();
    if (w == 0) {
#pragma unroll
      for (int k = 0; k < kAdjParts; ++k) v[k] = l < nw ? sh[k][l] : 0.0;
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {  // at most 8 warps
#pragma unroll
        for (int k = 0; k < kAdjParts; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
      }
    }
  };
  double v[kAdjParts];
#pragma unroll
  for (int k = 0; k < kAdjParts; ++k) v[k] = acc[k];
  reduce(v);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < kAdjParts; ++k) part[kAdjParts * (size_t)blockIdx.x + k] = v[k];
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
#pragma unroll
  for (int k = 0; k < kAdjParts; ++k) v[k] = 0.0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) {
#pragma unroll
    for (int k = 0; k < kAdjParts; ++k) v[k] += __ldcg(part + kAdjParts * (size_t)b + k);
  }
  reduce(v);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < kAdjParts; ++k) sums[k] = v[k];
    if (out.gth) {  // gth[0] += g0 q[0] + g4 q[4], gth[1] += g1 q[1] + g3 q[3]
      out.gth[0] += out.g0 * v[0] + out.g4 * v[4];
      out.gth[1] += out.g1 * v[1] + out.g3 * v[3];
    }
    *ticket = 0u;
  }
}

template <bool MIXED, bool WHOLE, bool FO>
__device__ __forceinline__ void adjoint_tile_compute(const TileShared& S, const unsigned char* buf, const TileLayout& L,
                                                     const uint2* __restrict__ rows, const uint16_t* __restrict__ ent,
                                                     const LJConst& c, const Geom& g, const dvec4* __restrict__ w,
                                                     const float4* __restrict__ wf, const AdjointOut& out,
                                                     int32_t* __restrict__ status, double* acc, int list_cap) {
  const void* sh_pos = buf + L.pos;
  const int* sh_gid = (const int*)(buf + L.gid);
  const uint2* s_rows = (const uint2*)(buf + L.rows);
  const uint16_t* s_ent = (const uint16_t*)(buf + L.ent);
  const int lane = threadIdx.x & (kAdjLanes - 1);
  const int grp = threadIdx.x / kAdjLanes;
  constexpr int kGroups = kTileThreads / kAdjLanes;
  const double e4 = 4.0 * c.eps, inv_sig = c.inv_sigma, c2s = c.c2s;
  const int n_own = S.own1 - S.own0;
  for (int o = grp; __any_sync(0xffffffffu, o < n_own); o += kGroups) {
    const bool valid = o < n_own;
    double h[3] = {0.0, 0.0, 0.0}, f[3] = {0.0, 0.0, 0.0}, q[kAdjParts] = {0.0, 0.0, 0.0, 0.0, 0.0};
    float ah[3] = {0.f, 0.f, 0.f}, af[3] = {0.f, 0.f, 0.f}, aq[4] = {0.f, 0.f, 0.f, 0.f};
    int gi = 0;
    if (valid) {
      const int l = S.own0 + o;
      gi = S.gown0 + o;
      uint2 row;
      const uint16_t* el;
      if (WHOLE) {
        row = rows[gi];
        el = ent;
      } else {
        row = s_rows[S.row_off + o];
        row.x -= S.list_base;
        el = row.x + row.y <= (unsigned)list_cap ? s_ent : ent + S.list_base;  // the end of a long segment stays in HBM
        if (row.x + row.y > S.list_len) {
          if (lane == 0) atomicOr(status, LJ_ST_LIST_OVERFLOW);
          row.y = 0;
        }
      }
      if (MIXED) {
        const uint4 qi = ((const uint4*)sh_pos)[l];
        const float e4f = c.e4, sig2f = c.sig2f, c2sf = c.c2sf, rc2f = c.rc2f, c0f = c.c0f, isgf = c.inv_sigmaf;
        const float4 wif = wf[gi];  // the FP32 copy of w (no conversions per pair)
        const float wx = wif.x, wy = wif.y, wz = wif.z;
        for (unsigned e = lane; e < row.y; e += kAdjLanes) {
          const int j = el[row.x + e];
          const uint4 qj = ((const uint4*)sh_pos)[j];
          // differences in sigma units: the integer difference in units of u, converted once and
          // scaled by u (a power of two: exact)
          const float dx = qd<WHOLE>(qj.x, qi.x, g) * g.qu, dy = qd<WHOLE>(qj.y, qi.y, g) * g.qu,
                      dz = qd<WHOLE>(qj.z, qi.z, g) * g.qu;
          const float s2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
          if (!(s2 < rc2f)) continue;
          const float4 wj = wf[qj.w];
          const float is = rcp_nr(s2);
          const float a = sig2f * is, a3 = a * a * a, a6 = a3 * a3;
          const float u = e4f * (a6 - a3 + c2sf * s2 + c0f);
          const float u1 = e4f * (is * (3.0f * a3 - 6.0f * a6) + c2sf);
          const float u2 = e4f * is * is * (42.0f * a6 - 12.0f * a3);
          const float dus = e4f * isgf * (12.0f * a6 - 6.0f * a3 - 2.0f * c2sf * s2);
          const float du1s = e4f * isgf * (is * (18.0f * a3 - 72.0f * a6) - 2.0f * c2sf);
          const float dwx = wx - wj.x, dwy = wy - wj.y, dwz = wz - wj.z;
          const float ddw = dx * dwx + dy * dwy + dz * dwz;
          const float t1 = 2.0f * u1, t2 = 4.0f * u2 * ddw;
          ah[0] += t1 * dwx + t2 * dx;
          ah[1] += t1 * dwy + t2 * dy;
          ah[2] += t1 * dwz + t2 * dz;
          if (FO) {
            af[0] += t1 * dx;
            af[1] += t1 * dy;
            af[2] += t1 * dz;
          }
          const float wd = wx * dx + wy * dy + wz * dz;
          aq[0] += t1 * wd;
          aq[1] += 2.0f * du1s * wd;
          aq[2] += 0.5f * u;
          aq[3] += 0.5f * dus;
        }
      } else {
        const dvec4 wi = w[gi];
        const dvec4 qi = ((const dvec4*)sh_pos)[l];
        for (unsigned e = lane; e < row.y; e += kAdjLanes) {
          const int j = el[row.x + e];
          const dvec4 qj = ((const dvec4*)sh_pos)[j];  // its image already in place (tiles)
          double dx = qj.x - qi.x, dy = qj.y - qi.y, dz = qj.z - qi.z;
          if (WHOLE) {
            dx = fma(-rint(dx * g.inv_L64), g.L, dx);
            dy = fma(-rint(dy * g.inv_L64), g.L, dy);
            dz = fma(-rint(dz * g.inv_L64), g.L, dz);
          }
          const double s2 = fma(dx, dx, fma(dy, dy, dz * dz));
          if (!(s2 < c.rc2)) continue;
          const dvec4 wj = w[sh_gid[j]];
          const double is = rcp_nr64(s2);
          const double a = c.sig2 * is, a3 = a * a * a, a6 = a3 * a3;
          const double u = e4 * (a6 - a3 + c2s * s2 + c.c0);
          const double u1 = e4 * (is * (3.0 * a3 - 6.0 * a6) + c2s);
          const double u2 = e4 * is * is * (42.0 * a6 - 12.0 * a3);
          const double dus = e4 * inv_sig * (12.0 * a6 - 6.0 * a3 - 2.0 * c2s * s2);
          const double du1s = e4 * inv_sig * (is * (18.0 * a3 - 72.0 * a6) - 2.0 * c2s);
          const double dwx = wi.x - wj.x, dwy = wi.y - wj.y, dwz = wi.z - wj.z;
          const double ddw = dx * dwx + dy * dwy + dz * dwz;
          const double t1 = 2.0 * u1, t2 = 4.0 * u2 * ddw;
          h[0] += t1 * dwx + t2 * dx;
          h[1] += t1 * dwy + t2 * dy;
          h[2] += t1 * dwz + t2 * dz;
          f[0] += t1 * dx;
          f[1] += t1 * dy;
          f[2] += t1 * dz;
          const double wd = wi.x * dx + wi.y * dy + wi.z * dz;
          q[0] += t1 * wd;
          q[1] += 2.0 * du1s * wd;
          q[2] += 0.5 * u;
          q[3] += 0.5 * dus;
          q[4] += 0.5 * u;
        }
      }
    }
    if (MIXED) {  // the group's lanes reduce in FP32; one lane converts and accumulates in FP64
      for (int k = 0; k < 3; ++k) {
        ah[k] = gsum<kAdjLanes>(ah[k]);
        if (FO) af[k] = gsum<kAdjLanes>(af[k]);
      }
      for (int k = 0; k < 4; ++k) aq[k] = gsum<kAdjLanes>(aq[k]);
      if (valid && lane == 0) {
        adjoint_row(out, gi, ah[0], ah[1], ah[2], af[0], af[1], af[2]);
        for (int k = 0; k < 4; ++k) acc[k] += f32_to_f64(aq[k]);  // (integer conversions: no FP64 slots)
      }
    } else {
      for (int k = 0; k < 3; ++k) {
        h[k] = gsum<kAdjLanes>(h[k]);
        f[k] = gsum<kAdjLanes>(f[k]);
      }
      if (valid && lane == 0) {
        adjoint_row(out, gi, h[0], h[1], h[2], f[0], f[1], f[2]);
      }
      for (int k = 0; k < kAdjParts; ++k) acc[k] += q[k];
    }
  }
}

// Bound by the latency of the gather of w (16 bytes a pair from L2) and by issue, so the mixed form runs four
// CTAs per SM (64 registers, FP32 sums of the parameter derivatives, forces only where they are wanted):
// 1,048,576 particles, rho = 0.5, r_c + margin 3.0: 570 us with two CTAs, 371 with three, 340 with four.
template <bool MIXED, bool WHOLE, bool FO>
__global__ void __launch_bounds__(kTileThreads, MIXED ? 4 : 2)
    k_adjoint_tile(const void* __restrict__ pos, const uint32_t* __restrict__ cs, int64_t N, Geom g, TileArgs ta,
                   LJConst c, const uint2* __restrict__ rows,
                   const uint2* __restrict__ tile_list, const uint16_t* __restrict__ ent,
                   const dvec4* __restrict__ w, const float4* __restrict__ wf, AdjointOut out,
                   double* __restrict__ part, unsigned int* __restrict__ ticket, double* __restrict__ sums,
                   int32_t* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ TileShared S;
  __shared__ __align__(8) uint64_t bar;
  const TileLayout L = tile_layout(ta, MIXED, true, !MIXED);
  double acc[kAdjParts] = {0.0, 0.0, 0.0, 0.0, 0.0};
  if (WHOLE) {
    if (blockIdx.x == 0) {
      stage_whole<MIXED, !MIXED>(N, pos, S, smem, L);
      __syncthreads();
      adjoint_tile_compute<MIXED, true, FO>(S, smem, L, rows, ent, c, g, w, wf, out, status, acc, ta.list_cap);
    }
  } else {
    if (threadIdx.x == 0) {
      mbar_init(&bar, 1);
      fence_proxy_async_smem();
    }
    __syncthreads();
    uint32_t ph = 0;
    for (int64_t t = blockIdx.x; t < ta.ntiles; t += gridDim.x) {
      const bool ok = force_tile_prepare(tile_info(t, ta), t, ta, cs, tile_list, S, status);
      if (ok) {
        const TileInfo ti = tile_info(t, ta);
        stage_issue<MIXED, true>(ti, ta, pos, rows, ent, S, smem, L, &bar);
        if (!stage_finish<MIXED, true>(ti, ta, g, S, smem, L, &bar, ph, !MIXED, status)) return;
        adjoint_tile_compute<MIXED, false, FO>(S, smem, L, rows, ent, c, g, w, wf, out, status, acc, ta.list_cap);
      }
      __syncthreads();
    }
  }
  if (MIXED) acc[4] = acc[2];  // both are PE
  adjoint_finish(acc, out, part, ticket, sums);
}

// ---------------------------------------------------------------------------------------------
// The adjoint pass of the FP64 form by queues (tiles): pairs inside r_c only, in full warps.  The general
// kernel above walks every listed pair with four threads a key, of which those outside r_c (42 %) idle
// through the others' FP64 operations.  FO: the forces are wanted too.  (In the mixed form queues lose:
// 613 us against 490 at 1,048,576 particles, as filling and draining them costs more than the idle lanes.)
//
// With A = sigma^6 ri6, t1 = 2 u' is the force's own coefficient and k2 = 4 u''; as the pair
// energy depends on s / sigma^2 alone, 2 du'/dsigma = -(2 / sigma) (t1 + k2 s / 2), and as every pair is
// visited from both sides with d of either sign, the sums of w . F and w . dF/dsigma are half those of
// t1 d . dw and of -(2 / sigma) (t1 + k2 s / 2) d . dw; PE and dPE/dsigma come from the sums of r^-6, r^-12
// and r^2: 35 FP64 operations a pair (38 with the forces) against about 65.
template <bool FO>
__global__ void __launch_bounds__(kDpThreads, 3)
    k_adjoint_dp(const dvec4* __restrict__ pos, const uint32_t* __restrict__ cs, Geom g, TileArgs ta, LJConst c,
                 const uint2* __restrict__ rows, const uint2* __restrict__ tile_list, const uint16_t* __restrict__ ent,
                 const dvec4* __restrict__ w, AdjointOut out, double* __restrict__ part,
                 unsigned int* __restrict__ ticket, double* __restrict__ sums, int32_t* __restrict__ status) {
  constexpr int NACC = FO ? 6 : 3;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ TileShared S;
  __shared__ __align__(8) uint64_t bar;
  const DpLayout D = dp_layout<NACC, false>(ta);
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_proxy_async_smem();
  }
  __syncthreads();
  const double sig6 = c.sig2 * c.sig2 * c.sig2, sig12 = sig6 * sig6;
  const double rc2 = c.rc2, f8c2 = 8.0 * c.eps * c.c2s, f24s = 24.0 * c.eps * sig6, f48s = 48.0 * c.eps * sig12;
  const double k672 = 672.0 * c.eps * sig12, k192 = 192.0 * c.eps * sig6;
  double q0 = 0.0, q1 = 0.0, s6 = 0.0, s12 = 0.0, s2 = 0.0, npairs = 0.0;
  int np = 0;
  uint32_t ph = 0;
  const dvec4* sp = (const dvec4*)(smem + D.L.pos);
  const uint4* sq = (const uint4*)(smem + D.xq);
  struct Key {
    dvec4 x, w;
  };
  for (int64_t t = blockIdx.x; t < ta.ntiles; t += gridDim.x) {
    const TileInfo ti = tile_info(t, ta);
    if (force_tile_prepare(ti, t, ta, cs, tile_list, S, status)) {
      stage_issue<false, true>(ti, ta, pos, rows, ent, S, smem, D.L, &bar);
      if (!dp_stage_finish(ti, ta, g, S, smem, D, &bar, ph, status)) return;
      queue_tile_pairs<NACC, false>(
          S, sq, (const uint2*)(smem + D.L.rows), ((DpWarp<NACC, false>*)(smem + D.warp))[threadIdx.x >> 5],
          (const uint16_t*)(smem + D.L.ent), ent + S.list_base, (unsigned)ta.list_cap, filter_cut2(c), status,
          [&](int o) { return Key{sp[S.own0 + o], w[S.gown0 + o]}; }, [&](int j) { return Key{sp[j], w[sq[j].w]}; },
          [&](const Key& k, const Key& j, double* acc) {
            const dvec4 &qj = j.x, &wj = j.w;
            const double dx = qj.x - k.x.x, dy = qj.y - k.x.y, dz = qj.z - k.x.z;
            const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
            if (!inside_rc(r2, rc2)) return;
            const double ri2 = rcp_cubic64(r2);
            const double ri4 = ri2 * ri2, ri6 = ri4 * ri2, ri8 = ri4 * ri4;
            const double t1 = fma(ri8, fma(-f48s, ri6, f24s), f8c2);
            const double k2 = (ri8 * ri2) * fma(k672, ri6, -k192);
            const double ux = k.w.x - wj.x, uy = k.w.y - wj.y, uz = k.w.z - wj.z;
            const double ddw = fma(dx, ux, fma(dy, uy, dz * uz));
            const double t2 = k2 * ddw;
            acc[0] = fma(t1, ux, fma(t2, dx, acc[0]));
            acc[1] = fma(t1, uy, fma(t2, dy, acc[1]));
            acc[2] = fma(t1, uz, fma(t2, dz, acc[2]));
            if (FO) {
              acc[NACC - 3] = fma(t1, dx, acc[NACC - 3]);
              acc[NACC - 2] = fma(t1, dy, acc[NACC - 2]);
              acc[NACC - 1] = fma(t1, dz, acc[NACC - 1]);
            }
            q0 = fma(t1, ddw, q0);
            q1 = fma(t2, r2, q1);
            s6 += ri6;
            s12 = fma(ri6, ri6, s12);
            s2 += r2;
            ++np;
          },
          [&](int o, const double* a) {
            adjoint_row(out, S.gown0 + o, a[0], a[1], a[2], FO ? a[NACC - 3] : 0.0, FO ? a[NACC - 2] : 0.0,
                        FO ? a[NACC - 1] : 0.0);
          });
      npairs += (double)np;
      np = 0;
    }
    __syncthreads();
  }
  double acc[kAdjParts];
  acc[0] = 0.5 * q0;
  acc[1] = -c.inv_sigma * fma(0.5, q1, q0);
  acc[4] = 2.0 * c.eps * fma(sig12, s12, fma(-sig6, s6, fma(c.c2s, s2, c.c0 * npairs)));
  acc[2] = acc[4];
  acc[3] = 2.0 * c.eps * c.inv_sigma * fma(12.0 * sig12, s12, fma(-6.0 * sig6, s6, -2.0 * c.c2s * s2));
  adjoint_finish(acc, out, part, ticket, sums);
}

size_t adjoint_smem_bytes(const TileArgs& ta, int precision) {
  return align16(tile_layout(ta, precision == LJ_MIXED, true, precision != LJ_MIXED).total);
}

// Fits the queues beside the staged FP64 tile, giving up staged list entries for them if need be.
static bool adjoint_dp_fits(TileArgs& ta) {
  int dev = 0, smem_max = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  TileArgs tz = ta;
  tz.list_cap = 0;
  // 3 KB: static shared memory (bookkeeping and final sums)
  const int64_t room = ((int64_t)smem_max - 3072 - (int64_t)dp_layout<6, false>(tz).total) / 2 - 8;
  if (ta.whole || room < 0) return false;
  ta.list_cap = (int32_t)(std::min<int64_t>(ta.list_cap, room) & ~(int64_t)7);
  return true;
}

int launch_adjoint_tile(int precision, const void* pos, const uint32_t* cs, int64_t N, Geom g, TileArgs ta, LJConst c,
                        const uint2* rows, const uint2* tile_list, const uint16_t* ent, const void* w,
                        const float4* wf, const AdjointOut& out, double* part, unsigned int* ticket, double* sums,
                        int32_t* status, cudaStream_t s) {
  const bool fo = out.fo != nullptr || out.a != 0.0;
  const bool mixed = precision == LJ_MIXED;
  TileArgs tq = ta;
  if (!mixed && adjoint_dp_fits(tq)) {
    int grid = 1;
#define LJ_ADJ_DP(FO, NACC)                                                                                          \
  do {                                                                                                               \
    const size_t sm_ = dp_layout<NACC, false>(tq).total;                                                             \
    set_smem(k_adjoint_dp<FO>, sm_);                                                                                 \
    grid = tile_grid(tq, resident_per_sm(k_adjoint_dp<FO>, kDpThreads, sm_));                                        \
    k_adjoint_dp<FO><<<grid, kDpThreads, sm_, s>>>((const dvec4*)pos, cs, g, tq, c, rows, tile_list, ent,            \
                                                   (const dvec4*)w, out, part, ticket, sums, status);                \
  } while (0)
    if (fo) LJ_ADJ_DP(true, 6);
    else LJ_ADJ_DP(false, 3);
#undef LJ_ADJ_DP
    return grid;
  }
  if (mixed && !ta.whole) {
    // four CTAs per SM if that still stages three quarters of the longest list segment; its end is read from
    // L2, which costs less than the fourth CTA gives (1 KB reserved and 2.5 KB static shared memory per CTA)
    int dev = 0, smem_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    TileArgs tz = ta;
    tz.list_cap = 0;
    const int64_t cap = ((int64_t)smem_sm / 4 - 3584 - (int64_t)adjoint_smem_bytes(tz, precision)) / 2 & ~(int64_t)7;
    if (4 * cap >= 3 * (int64_t)ta.max_list) ta.list_cap = (int32_t)std::min<int64_t>(ta.list_cap, cap);
  }
  const size_t sm = adjoint_smem_bytes(ta, precision);
  int grid = 1;
#define LJ_ADJ_LAUNCH_FO(M, W, FO)                                                                                   \
  do {                                                                                                               \
    set_smem(k_adjoint_tile<M, W, FO>, sm);                                                                          \
    grid = tile_grid(ta, resident_per_sm(k_adjoint_tile<M, W, FO>, kTileThreads, sm));                               \
    k_adjoint_tile<M, W, FO><<<grid, kTileThreads, sm, s>>>(pos, cs, N, g, ta, c, rows, tile_list, ent, (const dvec4*)w, \
                                                        wf, out, part, ticket, sums, status);                        \
  } while (0)
#define LJ_ADJ_LAUNCH(M, W)                  \
  do {                                       \
    if (fo) LJ_ADJ_LAUNCH_FO(M, W, true);    \
    else LJ_ADJ_LAUNCH_FO(M, W, false);      \
  } while (0)
  if (mixed) {
    if (ta.whole) LJ_ADJ_LAUNCH(true, true);
    else LJ_ADJ_LAUNCH(true, false);
  } else {
    if (ta.whole) LJ_ADJ_LAUNCH(false, true);
    else LJ_ADJ_LAUNCH(false, false);
  }
#undef LJ_ADJ_LAUNCH
#undef LJ_ADJ_LAUNCH_FO
  return grid;
}

int set_wait_budget_adjoint(long long cycles) { return set_unit_wait_budget(cycles); }

}  // namespace ljmd
