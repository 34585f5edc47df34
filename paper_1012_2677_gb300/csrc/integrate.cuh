// One particle's velocity-Verlet step, shared by the integrator and the force kernel that takes the step.
#pragma once

#include "common.cuh"

namespace ljmd {

// One particle's inputs to the integrator: force, velocity, position and (when the position copy is
// rewritten) the displacement reference.  F_L2: the force was written by other threads of the launch.
template <bool MIXED>
struct IntegrateIn;
template <>
struct IntegrateIn<true> {
  float4 f;
  uint4 r;
  double v[3], x[3];
};
template <>
struct IntegrateIn<false> {
  dvec4 f, r;
  double v[3], x[3];
};

template <bool MIXED, bool F_L2 = false>
__device__ __forceinline__ void integrate_load(IntegrateIn<MIXED>& in, const double* __restrict__ x,
                                               const double* __restrict__ v, const void* __restrict__ fptr,
                                               const void* __restrict__ refp, int64_t N, int64_t i, int shadow) {
  if constexpr (MIXED) {
    in.f = F_L2 ? __ldcg((const float4*)fptr + i) : ((const float4*)fptr)[i];
    if (shadow) in.r = ((const uint4*)refp)[i];
  } else {
    in.f = ((const dvec4*)fptr)[i];
    if (shadow) in.r = ((const dvec4*)refp)[i];
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    in.v[k] = v[k * N + i];
    in.x[k] = x[k * N + i];
  }
}

// What a thread sums over its particles.
struct IntegrateAcc {
  double ke = 0.0;
  float d2max = 0.0f, v2max = 0.0f;
  bool bad = false;
};

// The fixed-point coordinate floor(x / u + 1/2) as fixq gives it, by one operation of the FP64 pipe: with
// 1.5 2^51 added, rounding down leaves the half units in the significand's low bits.
__device__ __forceinline__ uint32_t fixq_fma(double x, double scale) {
  return (uint32_t)((unsigned long long)__double_as_longlong(__fma_rd(x, scale, 3377699720527872.0 + 0.5)) >> 1);
}

// HW: conversions (mixed form) by the FP64 pipe, for a kernel that is bound by issue and leaves that pipe idle.
template <bool MIXED, bool HW = false>
__device__ __forceinline__ void integrate_one(const IntegrateIn<MIXED>& in, const IntegrateArgs& a, double* __restrict__ x,
                                              double* __restrict__ v, void* __restrict__ pos, int64_t N, int64_t i,
                                              IntegrateAcc& acc) {
  const float qu = __int_as_float((127 - a.qk) << 23);  // u = 2^-qk
  const bool kick = !is_zero_d(a.kk), drift = !is_zero_d(a.dt);
  double F[3];
  float Ff[3] = {0.0f, 0.0f, 0.0f};
  if constexpr (MIXED) {
    const float4 f = in.f;
    Ff[0] = f.x;
    Ff[1] = f.y;
    Ff[2] = f.z;
    F[0] = HW ? (double)f.x : f32_to_f64(f.x);
    F[1] = HW ? (double)f.y : f32_to_f64(f.y);
    F[2] = HW ? (double)f.z : f32_to_f64(f.z);
  } else {
    const dvec4 f = in.f;
    F[0] = f.x;
    F[1] = f.y;
    F[2] = f.z;
  }
  double xs[3];
  float ke_i = 0.0f, vd2 = 0.0f;
  double ke_d = 0.0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double vk = in.v[k];
    if (a.ke) {
      if (MIXED) {
        const float vf = fmaf(a.kpre_f, Ff[k], HW ? __double2float_rn(vk) : f64_to_f32(vk));
        ke_i = fmaf(vf, vf, ke_i);
      } else {
        const double vf = fma(a.kpre, F[k], vk);
        ke_d = fma(vf, vf, ke_d);
      }
    }
    if (kick) vk = fma(a.kk, F[k], vk);
    if (a.speed) {
      const float vs = MIXED && !HW ? f64_to_f32(vk) : (float)vk;
      vd2 = fmaf(vs, vs, vd2);
    }
    double xk = in.x[k];
    if (drift) xk = fma(a.dt, vk, xk);
    v[k * N + i] = vk;
    x[k * N + i] = xk;
    xs[k] = xk;
    acc.bad |= !finite_d(xk) || (!HW && !finite_d(vk));  // HW drifts: dt v makes the position as bad
  }
  if (a.ke) {
    if (MIXED) acc.ke += f32_to_f64(0.5f * ke_i);  // exact halving and conversion, one FP64 add
    else acc.ke += 0.5 * ke_d;
  }
  if (a.shadow) {
    // speed of the drift (the velocity that moved the particle this step), for the DUTC rule
    acc.v2max = fmaxf(acc.v2max, vd2);
    if constexpr (MIXED) {
      auto fix = [&](double v) {
        return HW ? fixq_fma(v, a.scale) : fixq(v, a.qk);
      };
      const uint4 q = make_uint4(fix(xs[0]), fix(xs[1]), fix(xs[2]), (uint32_t)i);
      ((uint4*)pos)[i] = q;
      // displacement since the list was built, from the records: exact integer differences
      // (within u of the FP64 ones), converted once and scaled by u
      const uint4 r = in.r;
      const float dx = qdiff(q.x, r.x) * qu, dy = qdiff(q.y, r.y) * qu, dz = qdiff(q.z, r.z) * qu;
      acc.d2max = fmaxf(acc.d2max, fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
    } else {
      ((dvec4*)pos)[i] = make_dvec4(xs[0], xs[1], xs[2], 0.0);
      const dvec4 r = in.r;
      const double dx = xs[0] - r.x, dy = xs[1] - r.y, dz = xs[2] - r.z;
      // rounded up to FP32, so the measured maximum never falls short of the FP64 value and the
      // margin/2 rule keeps its guarantee at the FP64 form's tight limit
      acc.d2max = fmaxf(acc.d2max, __double2float_ru(fma(dx, dx, fma(dy, dy, dz * dz))));
    }
  }
}

}  // namespace ljmd
