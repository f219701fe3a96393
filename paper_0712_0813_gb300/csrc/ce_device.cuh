// ce_device.cuh -- device-side building blocks shared by the step kernels:
// the model (potential and its derivatives), the block reduction of the
// global sums, and the scale-factor update done by the last block of a step.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "ce_internal.h"

namespace ce {

__device__ __forceinline__ float fmaT(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmaT(double a, double b, double c) { return fma(a, b, c); }

// Model V = phi^4/4 + sum_i (q_i/2) phi^2 chi_i^2 (program units) at one site:
// dV/df for each field and V itself.  g[0] = phi, g[i>0] = chi_i.
template <typename T, int NF>
__device__ __forceinline__ void model_dv(const T (&g)[NF], const T (&q)[3], T (&dv)[NF], T& vsite) {
  const T phi = g[0];
  const T phi2 = phi * phi;
  T cpl = T(0);  // sum_i q_i chi_i^2
#pragma unroll
  for (int i = 1; i < NF; ++i) cpl = fmaT(q[i - 1] * g[i], g[i], cpl);
  dv[0] = phi * fmaT(phi, phi, cpl);
#pragma unroll
  for (int i = 1; i < NF; ++i) dv[i] = q[i - 1] * phi2 * g[i];
  vsite = phi2 * fmaT(T(0.25), phi2, T(0.5) * cpl);
}

// 16 bytes of consecutive sites: VX = 16 / sizeof(T) values, one vector access
// (read-only path for loads, streaming stores).
template <typename T, int VX>
__device__ __forceinline__ void ldg16v(const T* p, T (&o)[VX]) {
  if constexpr (sizeof(T) == 4) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(p));
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
  } else {
    const double2 v = __ldg(reinterpret_cast<const double2*>(p));
    o[0] = v.x; o[1] = v.y;
  }
}
template <typename T, int VX>
__device__ __forceinline__ void stcs16v(T* p, const T (&o)[VX]) {
  if constexpr (sizeof(T) == 4) {
    __stcs(reinterpret_cast<float4*>(p), make_float4(o[0], o[1], o[2], o[3]));
  } else {
    __stcs(reinterpret_cast<double2*>(p), make_double2(o[0], o[1]));
  }
}

// A value at a 32-bit byte offset from a base that is the same for the whole warp: the
// base stays in uniform registers and the access needs no 64-bit address arithmetic.
template <typename T>
__device__ __forceinline__ T ldg_at(const T* base, uint32_t bytes) {
  return __ldg(reinterpret_cast<const T*>(reinterpret_cast<const char*>(base) + bytes));
}
template <typename T>
__device__ __forceinline__ void stcs_at(T* base, uint32_t bytes, T v) {
  __stcs(reinterpret_cast<T*>(reinterpret_cast<char*>(base) + bytes), v);
}

// One 16-byte group of the 1D step: VX = 16 / sizeof(T) consecutive sites
// starting at site s = k VX of a periodic 1D lattice of N sites (N a multiple
// of VX), all fields.  16-byte loads of the group's f and w, scalar loads of the
// two outer neighbours (the neighbouring groups' vectors already brought them
// into L1), each site's g = f + dd (w + c f) formed once per field, then
// w_out = v + kk (lap g - dV/df(g)) and f_out = g with 16-byte streaming stores.
// The per-site operations and their order are those of the generic kernel, so
// every 1D kernel built on this gives the same fields bit for bit.  Adds the
// group's sum of (g(x+1) - g(x))^2 and of V(g) to g2loc and vloc.
template <typename T, int NF>
__device__ __forceinline__ void step1d_group(const T* const (&f_in)[4], const T* const (&w_in)[4],
                                             T* const (&f_out)[4], T* const (&w_out)[4], int64_t N, int64_t k,
                                             T c, T dd, T kk, T idx2, const T (&q)[3], T& g2loc, T& vloc) {
  constexpr int VX = 16 / sizeof(T);
  const int64_t s = k * VX;
  const int64_t sl = (k == 0) ? N - 1 : s - 1;             // left neighbour of the first site
  const int64_t sr = (s + VX == N) ? 0 : s + VX;           // right neighbour of the last site
  T g[NF][VX + 2], v[NF][VX];   // g[i][1 + j] at site s + j; [0] and [VX + 1] the outer neighbours
#pragma unroll
  for (int i = 0; i < NF; ++i) {
    T f[VX], w[VX];
    ldg16v<T, VX>(f_in[i] + s, f);
    ldg16v<T, VX>(w_in[i] + s, w);
#pragma unroll
    for (int j = 0; j < VX; ++j) {
      v[i][j] = fmaT(c, f[j], w[j]);
      g[i][j + 1] = fmaT(dd, v[i][j], f[j]);
    }
    const T fl = __ldg(f_in[i] + sl), wl = __ldg(w_in[i] + sl);
    const T fr = __ldg(f_in[i] + sr), wr = __ldg(w_in[i] + sr);
    g[i][0] = fmaT(dd, fmaT(c, fl, wl), fl);
    g[i][VX + 1] = fmaT(dd, fmaT(c, fr, wr), fr);
  }
  T wo[NF][VX], fo[NF][VX];
#pragma unroll
  for (int j = 0; j < VX; ++j) {
    T gs[NF], lap[NF];
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      const T gc = g[i][j + 1], gp = g[i][j + 2], gm = g[i][j];
      T acc = T(0);
      acc += (gp + gm) - T(2) * gc;
      const T df = gp - gc;
      g2loc = fmaT(df, df, g2loc);
      lap[i] = acc * idx2;
      gs[i] = gc;
    }
    T dv[NF], vs;
    model_dv<T, NF>(gs, q, dv, vs);
    vloc += vs;
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      wo[i][j] = fmaT(kk, lap[i] - dv[i], v[i][j]);
      fo[i][j] = gs[i];
    }
  }
#pragma unroll
  for (int i = 0; i < NF; ++i) {
    stcs16v<T, VX>(w_out[i] + s, wo[i]);
    stcs16v<T, VX>(f_out[i] + s, fo[i]);
  }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ int64_t linear_block_id() {
  return (int64_t)blockIdx.x + (int64_t)gridDim.x * ((int64_t)blockIdx.y + (int64_t)gridDim.y * blockIdx.z);
}

__device__ __forceinline__ int64_t grid_blocks() {
  return (int64_t)gridDim.x * gridDim.y * gridDim.z;
}

// FP64 is scarce here: a warp instruction takes one of the SM's four FP64 pipes for
// 64 cycles, whether one lane needs it or 32, and its result as long (measured: add,
// multiply, FMA and conversion 64 each, division 554, square root 607).  So what
// runs once per block or per step is written for few FP64 instructions: the end of
// a block and of a launch below took ~6 us of a step, the launch gap ~2.

// hi + lo += x: the addition's rounding error (Knuth's TwoSum, exact) joins lo.  Intrinsics,
// which the compiler does not contract with a product that x may be: else what is added
// would depend on the code around.
__device__ __forceinline__ void add_to(float& hi, float& lo, float x) {
  const float s = __fadd_rn(hi, x);
  const float b = __fsub_rn(s, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(x, b)));
  hi = s;
}

// A sum kept as an unevaluated pair of floats (48 bits).
struct FloatPair {
  float hi, lo;
};
// Sum of the lanes' pairs (valid in lane 0; lanes of `width` only).
template <int WIDTH>
__device__ __forceinline__ void warp_sum_pair(FloatPair& x) {
#pragma unroll
  for (int o = WIDTH / 2; o > 0; o >>= 1) {
    x.lo += __shfl_down_sync(0xffffffffu, x.lo, o);
    add_to(x.hi, x.lo, __shfl_down_sync(0xffffffffu, x.hi, o));
  }
}

// A block's share of 2 G + 3 V from its threads' two-level FP32 sums g0 + g1 and
// v0 + v1 (fixed order, valid in thread 0).  The sums are combined and added as float
// pairs (the per-thread sums' own rounding stays what limits them): three FP64
// instructions a block; sums that would leave the range in which a pair holds 48 bits
// of them, or of their products, take FP64 throughout.
__device__ __forceinline__ double block_source(float g0, float g1, float v0, float v1, const SourceWeights& k) {
  __shared__ float2 part[32];
  __shared__ double wide[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = (blockDim.x + 31) >> 5;
  FloatPair t{g0, 0.f}, v{v0, 0.f};
  add_to(t.hi, t.lo, g1);
  add_to(v.hi, v.lo, v1);
  const float p = __fmul_rn(k.ratio, v.hi);
  t.lo += fmaf(k.ratio, v.hi, -p) + fmaf(k.ratio_lo, v.hi, k.ratio * v.lo);
  add_to(t.hi, t.lo, p);
  const float size = fabsf(t.hi);
  const bool fits = size < 0x1p100f && (size > 0x1p-90f || (t.hi == 0.f && v.hi == 0.f));
  warp_sum_pair<32>(t);
  if (lane == 0) part[warp] = make_float2(t.hi, t.lo);
  if (__syncthreads_or(!fits)) {
    const double q = warp_sum(fma((double)v0 + (double)v1, k.wv, ((double)g0 + (double)g1) * k.wg));
    if (lane == 0) wide[warp] = q;
    __syncthreads();
    double sum = 0.0;
    if (threadIdx.x == 0)
      for (int w = 0; w < nwarps; ++w) sum += wide[w];
    return sum;
  }
  double q = 0.0;
  if (warp == 0) {
    const float2 x = lane < nwarps ? part[lane] : make_float2(0.f, 0.f);
    FloatPair s{x.x, x.y};
    warp_sum_pair<32>(s);
    if (lane == 0) q = ((double)s.hi + (double)s.lo) * k.wg;
  }
  return q;
}

// Sum over the block of one FP64 value, fixed order, valid in thread 0.
__device__ __forceinline__ double block_sum(double a) {
  __shared__ double part[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = (blockDim.x + 31) >> 5;
  a = warp_sum(a);
  if (lane == 0) part[warp] = a;
  __syncthreads();
  if (warp == 0) {
    a = lane < nwarps ? part[lane] : 0.0;
    for (int o = nwarps > 16 ? 16 : (nwarps > 8 ? 8 : 4); o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
  }
  return a;
}

// The update (ce_source.h) by one thread; a source that leaves no real a' is latched.
__device__ __forceinline__ void scale_factor_update(const ScaleAhead& s, DevScalars& out, double source, double inv_dt,
                                                    int* status) {
  if (!scale_update(s, out, source, inv_dt)) atomicCAS(status, CE_OK, CE_ENONFINITE);
}

// End of a step launch: publish this block's share of 2 G + 3 V (in thread 0), and
// let the last block to finish combine all blocks' shares (fixed order over block
// index) and advance a, a', a''.  No block ever waits for another: the last
// arriving block does the work.
template <typename T>
__device__ __forceinline__ void finish_step(const StepArgs<T>& p, double share) {
  __shared__ int am_last;
  const int64_t nb = grid_blocks();
  if (threadIdx.x == 0) {
    p.partials[linear_block_id()] = share;
    __threadfence();
    const unsigned int prev = atomicAdd(p.counter, 1u);
    am_last = (prev == (unsigned int)(nb - 1));
  }
  __syncthreads();
  if (!am_last) return;
  __threadfence();
  ScaleAhead ahead;
  if (threadIdx.x == 0) ahead = scale_ahead(*p.sc_in, p.dt, p.kappa2);
  double sum = 0.0;
  for (int64_t j = threadIdx.x; j < nb; j += blockDim.x) sum += __ldcg(p.partials + j);
  sum = block_sum(sum);
  if (threadIdx.x == 0) {
    DevScalars out;
    scale_factor_update(ahead, out, sum, p.inv_dt, p.status);
    *p.sc_out = out;
    *p.counter = 0u;
  }
}

// The same from the threads' FP32 sums of (df)^2 and V, in two levels each.
__device__ __forceinline__ void finish_step_sums(const StepArgs<float>& p, float g0, float g1, float v0, float v1) {
  finish_step(p, block_source(g0, g1, v0, v1, p.source));
}
// And from FP64 sums.
__device__ __forceinline__ void finish_step_sums(const StepArgs<double>& p, double g0, double g1, double v0, double v1) {
  finish_step(p, block_sum(fma(v0 + v1, p.source.wv, (g0 + g1) * p.source.wg)));
}

}  // namespace ce
