// Velocity-Verlet (the benchmark's second-order symplectic integrator, Sec. 4.5), fused:
//
//   v_full = v + kpre F          (completes the previous step; its kinetic energy is taken)
//   v     <- v + (kpre + kpost) F (the first half-kick of the next step folded in)
//   x     <- x + dt v             (drift)
//
// then the force kernel's copy of the positions is rewritten (mixed form: the 32-bit fixed-point
// records, X = round(x_state / u) mod 2^32 with u = 2^-qk and the sorted index in w; FP64 form: a
// dvec4 copy) and the displacement since the last list construction is reduced (device-wide max)
// for the margin/2 validity rule.
// State x, v is FP64 (positions stored as offset + x).  Per component the FP64 pipe does two
// FMAs; the kinetic energy of the mixed form is taken in FP32 per particle and summed in FP64.
// In the mixed form every FP32 <-> FP64 conversion is done with integer operations (exact for
// FP32 -> FP64, rounded to nearest for FP64 -> FP32), which keeps the FP64 pipe for the seven
// operations per particle that need it.
#include "integrate.cuh"

namespace ljmd {

// Hint that the lines holding particle j's inputs be brought into L2 (one prefetch per stream; no
// registers are held for the data).
template <bool MIXED>
__device__ __forceinline__ void integrate_prefetch_l2(const double* x, const double* v, const void* fptr,
                                                      const void* refp, int64_t N, int64_t j, int shadow) {
  const void* f = MIXED ? (const void*)((const float4*)fptr + j) : (const void*)((const dvec4*)fptr + j);
  asm volatile("prefetch.global.L2 [%0];" ::"l"(f));
  if (shadow) {
    const void* r = MIXED ? (const void*)((const uint4*)refp + j) : (const void*)((const dvec4*)refp + j);
    asm volatile("prefetch.global.L2 [%0];" ::"l"(r));
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(v + k * N + j));
    asm volatile("prefetch.global.L2 [%0];" ::"l"(x + k * N + j));
  }
}

// The grid-stride loop is software-pipelined: the next particle's loads are issued before the
// FP64 kick and drift of the current one, so that the FP64 pipe (7 operations per particle at
// 1/64 of the FP32 rate) works while those loads are in flight instead of after them, and the lines
// of the particle kPrefetchAhead strides on are requested into L2, which keeps more of HBM's
// requests in flight than the registers of two particles per thread can.
constexpr int kPrefetchAhead = 2;

template <bool MIXED>
__global__ void __launch_bounds__(256) k_integrate(double* __restrict__ x, double* __restrict__ v,
                                                   const void* __restrict__ fptr, void* __restrict__ pos,
                                                   const void* __restrict__ refp, int64_t N, IntegrateArgs a,
                                                   double* __restrict__ ke_part, uint32_t* __restrict__ dmax_bits,
                                                   int32_t* __restrict__ status, StepFinish fin,
                                                   const int* __restrict__ skip) {
  if (skip && *skip) return;  // a device-decided run stopped before this step
  IntegrateAcc acc;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  IntegrateIn<MIXED> cur = {};
  if (i < N) integrate_load<MIXED>(cur, x, v, fptr, refp, N, i, a.shadow);
  for (; i < N; i += stride) {
    IntegrateIn<MIXED> nxt = {};
    if (i + stride < N) integrate_load<MIXED>(nxt, x, v, fptr, refp, N, i + stride, a.shadow);
    if (i + kPrefetchAhead * stride < N)
      integrate_prefetch_l2<MIXED>(x, v, fptr, refp, N, i + kPrefetchAhead * stride, a.shadow);
    integrate_one<MIXED>(cur, a, x, v, pos, N, i, acc);
    cur = nxt;
  }
  double ke_acc = acc.ke;
  float d2max = acc.d2max, v2max = acc.v2max;
  if (acc.bad) atomicOr(status, LJ_ST_NONFINITE);
  __shared__ double sh[32];
  __shared__ float shf[32];
  if (a.ke) {
    const double tk = block_sum(ke_acc, sh);
    if (threadIdx.x == 0) ke_part[blockIdx.x] = tk;
  }
  if (a.shadow && !a.speed) {
    const float m = block_max(d2max, shf);
    if (threadIdx.x == 0) atomicMax(dmax_bits, __float_as_uint(m));
  } else if (a.shadow) {  // both maxima in one pass over the warps
    __shared__ float shv[32];
    d2max = warp_max(d2max);
    v2max = warp_max(v2max);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) {
      shf[w] = d2max;
      shv[w] = v2max;
    }
    __syncthreads();
    if (w == 0) {
      const bool in = l < (int)(blockDim.x >> 5);
      const float md = warp_max(in ? shf[l] : 0.0f), mv = warp_max(in ? shv[l] : 0.0f);
      if (l == 0) {
        atomicMax(dmax_bits, __float_as_uint(md));
        atomicMax(dmax_bits + 1, __float_as_uint(mv));
      }
    }
  }
  if (fin.ticket) step_finish(fin, ke_part, dmax_bits);
}

// Block shape: 256-thread blocks of one resident wave (at most red_blocks(N)), so that the grid-stride
// loop ends in step on every SM; for a system too small to give every SM a block, narrower blocks
// (down to one warp) spread the particles over the SMs, each of whose FP64 pipes takes 1/64 of the
// FP32 rate.
template <bool MIXED>
static void integrate_shape(int64_t N, int& blocks, int& threads) {
  static int per_sm = 0, sms = 0;
  if (per_sm == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_integrate<MIXED>, kRedThreads, 0) != cudaSuccess ||
        per_sm < 1)
      per_sm = 1;
  }
  threads = kRedThreads;
  while (threads > 32 && (N + threads - 1) / threads < sms) threads >>= 1;
  if (threads == kRedThreads) {
    const int b = red_blocks(N);
    blocks = b < per_sm * sms ? b : per_sm * sms;
  } else {
    const int64_t b = (N + threads - 1) / threads;  // below 2 sms: within the partial arrays
    blocks = (int)(b < 1 ? 1 : b);
  }
}

int launch_integrate(int precision, double* x, double* v, const void* f, void* pos, const void* ref, int64_t N,
                     IntegrateArgs a, double* ke_part, uint32_t* dmax_bits, int32_t* status, StepFinish fin,
                     cudaStream_t s, const int* skip) {
  int blocks = 1, threads = kRedThreads;
  a = integrate_prepare(a);
  if (precision == LJ_MIXED) {
    integrate_shape<true>(N, blocks, threads);
    k_integrate<true><<<blocks, threads, 0, s>>>(x, v, f, pos, ref, N, a, ke_part, dmax_bits, status, fin, skip);
  } else {
    integrate_shape<false>(N, blocks, threads);
    k_integrate<false><<<blocks, threads, 0, s>>>(x, v, f, pos, ref, N, a, ke_part, dmax_bits, status, fin, skip);
  }
  return blocks;
}

// Position copies for the force and list kernels from the FP64 state (no integration): the FP32
// hi parts always, with the sorted index in w (the list construction filters on them in both
// forms); for the mixed form the fixed-point records, for FP64 the dvec4 copy; and the
// displacement reference (the records for mixed, the dvec4 for FP64) if ref != NULL.
__global__ void k_shadow(const double* __restrict__ x, int64_t N, int mixed, int qk, float4* __restrict__ hi,
                         uint4* __restrict__ xq, dvec4* __restrict__ pos64, void* __restrict__ ref,
                         const int* __restrict__ pred) {
  if (pred && !*pred) return;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
    const double a = x[i], b = x[N + i], c = x[2 * N + i];
    float4 h;
    float unused;
    split_hi_lo(a, h.x, unused);
    split_hi_lo(b, h.y, unused);
    split_hi_lo(c, h.z, unused);
    h.w = __int_as_float((int)i);  // the sorted index, for the list construction
    hi[i] = h;
    if (mixed) {
      const uint4 q = make_uint4(fixq(a, qk), fixq(b, qk), fixq(c, qk), (uint32_t)i);
      xq[i] = q;
      if (ref) ((uint4*)ref)[i] = q;
    } else {
      pos64[i] = make_dvec4(a, b, c, 0.0);
      if (ref) ((dvec4*)ref)[i] = make_dvec4(a, b, c, 0.0);
    }
  }
}

void launch_shadow_all(const double* x, int64_t N, int mixed, int qk, float4* hi, uint4* xq, dvec4* pos64, void* ref,
                       cudaStream_t s, const int* pred) {
  k_shadow<<<stride_grid(N, 256, pred), 256, 0, s>>>(x, N, mixed, qk, hi, xq, pos64, ref, pred);
}

}  // namespace ljmd
