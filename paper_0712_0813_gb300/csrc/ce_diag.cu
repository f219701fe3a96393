// ce_diag.cu -- the diagnostics pass: kinetic, gradient and potential energies
// and the fields' moments in one sweep over f and w, reduced and turned into
// the outputs by the launch's last block (one launch per read-out).
//
// Per site (arXiv:0712.0813 Sec. II outputs; the synchronised velocity is
// that of site_u in ce_generic.cu):
//   v_half = w + c f;  v(t_n) = v_half - dt/2 (lap f - dV/df + s f)
//   a'(t_n) = a'_{n+1/2} - dt/2 a''_n;  u = v(t_n) - (a'(t_n)/a_n) f
// With raw_u (start-up input) u is w itself.
//
// The pass reads f and w once (2 NF x sizeof(T) per site).  For FP32 storage HBM
// bounds it, provided the FP64 pipe (two lanes per clock and SM: 64 cycles a warp
// instruction and scheduler) stays out of it: a thread's partials over at most 16
// sites (in FP32, on smaller lattices in float pairs: Partials) are added, with the
// addition's rounding error kept (add_to), to float pairs of 48 bits, which the lanes
// add the same way; only the warps' sums become FP64.  That flush, as a counter
// test inside the site loop, was if-converted into 9 conversions and 9 FP64
// additions a site (256^3, two fields: 606 us where the bytes take 40), and as a
// loop of its own still took 202 us, half of it the warps' FP64 shuffle sums.
// FP64 storage is bound by its FP64 arithmetic.
#include <algorithm>
#include <cstdint>

#include "ce_device.cuh"
#include "ce_internal.h"

namespace ce {
namespace {

constexpr int kDiagThreads = 256;
constexpr int kDiagWarps = kDiagThreads / 32;
constexpr int kFlush = 16;   // sites a thread sums in T before adding to its running sums

// How the lattice is cut into block tasks.  3D: a task is 32 x-sites by 8 rows
// (one per warp, so the y-neighbours of the inner rows hit L1) swept along a
// chunk of z; 2D: 256 x-sites swept along a chunk of y; 1D: 256 threads x 16
// sites, strided.  Along the sweep the neighbours stay in registers.  Chunks of 16
// (their end planes, read twice, hit L2), shorter where that leaves blocks without
// a task: there one thread's sweep is pure latency.  FP64, whose arithmetic costs more
// than its loads, takes 256 consecutive sites of a plane in 3D (no lanes idle past a
// row's end), chunks down to one site, and skips warps without sites: ce_energy
// with four fields at 33^3 took 64 us in 32 x 8 tiles and chunks of 4 (now 50; 48 before
// the sweeps, with a thread a site), 101^3 394 (275; 376), 1D 4099 68 in chunks of 16 (30;
// 34).  Warp strips with the y- and
// x-neighbours in registers and a plane of loads in flight (the column kernel's
// layout) need half the loads but 164 registers: 217 against 142 us at 256^3.
struct DiagTasks {
  int nx, ny;      // x-segments (2D, 3D), row groups (3D)
  int len;         // sites per task along the sweep
  int64_t count;
};

DiagTasks diag_tasks(int dims, bool f64, int64_t N, int64_t S, int blocks) {
  DiagTasks t{1, 1, kFlush, 0};
  const bool linear = dims == 3 && f64;
  if (linear) t.nx = (int)((N * N + kDiagThreads - 1) / kDiagThreads);
  else if (dims > 1) t.nx = (int)((N + (dims == 3 ? 31 : kDiagThreads - 1)) / (dims == 3 ? 32 : kDiagThreads));
  if (dims == 3 && !linear) t.ny = (int)((N + kDiagWarps - 1) / kDiagWarps);
  const int shortest = f64 ? 1 : (dims == 1 ? kFlush : 4);
  const int want = f64 ? blocks : blocks / 2;
  for (t.len = kFlush;; t.len /= 2) {
    t.count = dims == 1 ? (S + (int64_t)kDiagThreads * t.len - 1) / ((int64_t)kDiagThreads * t.len)
                        : (int64_t)t.nx * t.ny * ((N + t.len - 1) / t.len);
    if (t.count >= want || t.len == shortest) return t;
  }
}

// Per-launch scalars in the storage type.
template <typename T>
struct DiagScalars {
  T idx2, half_dt, c, h, sterm;
  T q[3];
};

template <typename T>
__device__ __forceinline__ DiagScalars<T> diag_scalars(const DiagArgs<T>& p) {
  DiagScalars<T> k;
  const DevScalars sc = *p.sc;
  k.idx2 = (T)p.inv_dx2;
  k.half_dt = (T)(0.5 * p.dt);
  k.c = (T)sc.c;
  k.h = (p.expansion && !p.raw_u) ? (T)((sc.ap - 0.5 * p.dt * sc.app) / sc.a) : T(0);
  k.sterm = (p.expansion && !p.raw_u) ? (T)sc.s : T(0);
#pragma unroll
  for (int i = 0; i < 3; ++i) k.q[i] = (T)p.q[i];
  return k;
}

// A thread's sums over the sites of a task, up to kFlush of them: in T, or in pairs of
// floats (FP32 lattices below kPairSites).  Few sites leave few sums for their rounding to
// average over: in plain FP32 V of 1D 65536 was off by 1.1e-9 where FP64 sums of the sites
// give 2.8e-10 and the pairs 2.3e-10.  Large lattices keep 16 sites in FP32 (256^3: V 3e-10
// either way, 138 us against 181 with pairs; 1D 2 M 49 us with, 44 without); the
// squares of a site's gradient are added before they join the sum, without which G was
// off by 1.6e-8 (3.2e-9).
constexpr int64_t kPairSites = 5000000;

template <typename T, int NV, bool PAIRS>
struct Partials {
  T v[NV];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int j = 0; j < NV; ++j) v[j] = T(0);
  }
  __device__ __forceinline__ void add(int j, T x) { v[j] += x; }
  __device__ __forceinline__ void add_product(int j, T x, T y) { v[j] = fmaT(x, y, v[j]); }
};
template <int NV>
struct Partials<float, NV, true> {
  float v[NV], lo[NV];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int j = 0; j < NV; ++j) v[j] = lo[j] = 0.f;
  }
  __device__ __forceinline__ void add(int j, float x) { add_to(v[j], lo[j], x); }
  __device__ __forceinline__ void add_product(int j, float x, float y) { add(j, x * y); }
};

// One site's terms added to part: [K_i (NF)][G_i (NF)][V][f_i - f_i(0) (NF)]
// [(f_i - f_i(0))^2 (NF)].  nb[d][0] / nb[d][1]: the neighbours at +e_d / -e_d.
template <bool PAIRS, typename T, int NF, int DIMS>
__device__ __forceinline__ void diag_site(const DiagScalars<T>& k, int raw_u, const T (&f)[NF], const T (&w)[NF],
                                          const T (&nb)[NF][DIMS][2], const T (&shift)[NF],
                                          Partials<T, 4 * NF + 1, PAIRS>& part) {
  T dv[NF], vs;
  model_dv<T, NF>(f, k.q, dv, vs);
  part.add(2 * NF, vs);
#pragma unroll
  for (int i = 0; i < NF; ++i) {
    T lap = T(0);
    if constexpr (sizeof(T) == 8) {   // fewer FP64 operations; its rounding is far below the sums'
      T sum = nb[i][0][0] + nb[i][0][1];
#pragma unroll
      for (int d = 1; d < DIMS; ++d) sum += nb[i][d][0] + nb[i][d][1];
      lap = fmaT(T(-2 * DIMS), f[i], sum);
    } else {
#pragma unroll
      for (int d = 0; d < DIMS; ++d) lap += (nb[i][d][0] + nb[i][d][1]) - T(2) * f[i];
    }
    if constexpr (sizeof(T) == 8) {
#pragma unroll
      for (int d = 0; d < DIMS; ++d) part.add_product(NF + i, nb[i][d][0] - f[i], nb[i][d][0] - f[i]);
    } else {
      T g2 = T(0);
#pragma unroll
      for (int d = 0; d < DIMS; ++d) {
        const T df = nb[i][d][0] - f[i];
        g2 = fmaT(df, df, g2);
      }
      part.add(NF + i, g2);
    }
    T u = w[i];
    if (!raw_u) {
      const T vh = fmaT(k.c, f[i], w[i]);
      const T F = fmaT(lap, k.idx2, -dv[i]) + k.sterm * f[i];
      u = fmaT(-k.half_dt, F, vh) - k.h * f[i];
    }
    part.add_product(i, T(0.5) * u, u);
    const T df = f[i] - shift[i];
    part.add(2 * NF + 1 + i, df);
    part.add_product(3 * NF + 1 + i, df, df);
  }
}

// A thread's running sums: FP64, or float pairs.  Partials of 2^100 and above,
// infinities and NaN would leave the pairs' range: they go to the block's FP64
// sums `big` in shared memory.
template <typename T, int NV>
struct RunningSums;
template <int NV>
struct RunningSums<double, NV> {
  double v[NV];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int j = 0; j < NV; ++j) v[j] = 0.0;
  }
  __device__ __forceinline__ void add(const Partials<double, NV, false>& part, double*) {
#pragma unroll
    for (int j = 0; j < NV; ++j) v[j] += part.v[j];
  }
  __device__ __forceinline__ double warp_total(int j) { return warp_sum(v[j]); }
};
template <int NV>
struct RunningSums<float, NV> {
  float hi[NV], lo[NV];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int j = 0; j < NV; ++j) hi[j] = lo[j] = 0.f;
  }
  template <bool PAIRS>
  __device__ __forceinline__ void add(const Partials<float, NV, PAIRS>& part, double* big) {
    bool fits = true;
#pragma unroll
    for (int j = 0; j < NV; ++j) fits = fits && fabsf(part.v[j]) < 0x1p100f;
    if (__all_sync(0xffffffffu, fits)) {   // every lane of the warp is here
#pragma unroll
      for (int j = 0; j < NV; ++j) {
        add_to(hi[j], lo[j], part.v[j]);
        if constexpr (PAIRS) lo[j] += part.lo[j];
      }
    } else {
#pragma unroll
      for (int j = 0; j < NV; ++j) {
        double x = part.v[j];
        if constexpr (PAIRS) x += isfinite(part.lo[j]) ? (double)part.lo[j] : 0.0;
        atomicAdd(big + j, x);
      }
    }
  }
  __device__ __forceinline__ double warp_total(int j) {
    float h = hi[j], l = lo[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      l += __shfl_down_sync(0xffffffffu, l, o);
      add_to(h, l, __shfl_down_sync(0xffffffffu, h, o));
    }
    return (threadIdx.x & 31) == 0 ? (double)h + (double)l : 0.0;
  }
};

// The launch's last block: combine the blocks' sums (warp k takes quantity k,
// k + 8, ...; lane l takes blocks l, l + 32, ..., then a fixed shuffle tree) and
// derive the outputs.
template <typename T, int NF>
__device__ __forceinline__ void diag_outputs(const DiagArgs<T>& p, int blocks) {
  constexpr int NV = 4 * NF + 1;
  __shared__ double tot[NV];
  const int lane = threadIdx.x & 31;
  for (int k = threadIdx.x >> 5; k < NV; k += kDiagWarps) {
    double t = 0.0;
#pragma unroll 4
    for (int b = lane; b < blocks; b += 32) t += __ldcg(p.partials + (int64_t)b * NV + k);
    t = warp_sum(t);
    if (lane == 0) tot[k] = t;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  double* r = p.aux->result;
  for (int k = 0; k < kResultLen; ++k) r[k] = 0.0;
  const double invS = 1.0 / (double)p.S;
  double K = 0.0, G = 0.0;
  for (int i = 0; i < NF; ++i) {
    r[R_K + i] = tot[i] * invS;
    r[R_G + i] = tot[NF + i] * (0.5 * p.inv_dx2) * invS;
    K += tot[i] * invS;
    G += tot[NF + i] * (0.5 * p.inv_dx2) * invS;
  }
  const double V = tot[2 * NF] * invS;
  const double E = K + G + V;
  r[R_V] = V;
  r[R_KTOT] = K;
  r[R_GTOT] = G;
  r[R_E] = E;
  const DevScalars s = *p.sc;
  const double ap_t = p.expansion ? s.ap - 0.5 * p.dt * s.app : 0.0;
  r[R_A] = p.expansion ? s.a : 1.0;
  r[R_AP] = ap_t;
  r[R_RESID] = p.expansion ? fabs(ap_t * ap_t / p.kappa2 - E) / E : 0.0;
  for (int i = 0; i < NF; ++i) {
    const double m1 = tot[2 * NF + 1 + i] * invS;   // <f - f(0)>
    const double m2 = tot[3 * NF + 1 + i] * invS;   // <(f - f(0))^2>
    r[R_MEAN + i] = m1 + (double)p.f[i][0];
    r[R_VAR + i] = m2 - m1 * m1;
  }
  if (!isfinite(E)) atomicCAS(&p.aux->status, CE_OK, CE_ENONFINITE);
}

// End of a launch: the block's sums (the first NS quantities; zero beyond), and in the
// last block the outputs.
template <typename T, int NF, int NS>
__device__ __forceinline__ void diag_finish(const DiagArgs<T>& p, RunningSums<T, NS>& acc, double* big) {
  constexpr int NV = 4 * NF + 1;
  __shared__ double red[kDiagWarps][NS];
  __shared__ int s_last;
#pragma unroll
  for (int j = 0; j < NS; ++j) {
    const double v = acc.warp_total(j);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][j] = v;
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    double t = 0.0;
    if (threadIdx.x < NS) {
      t = big[threadIdx.x];
      for (int w = 0; w < kDiagWarps; ++w) t += red[w][threadIdx.x];
    }
    p.partials[(int64_t)blockIdx.x * NV + threadIdx.x] = t;
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&p.aux->counter_diag, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  diag_outputs<T, NF>(p, gridDim.x);
  if (threadIdx.x == 0) p.aux->counter_diag = 0u;
}

template <typename T, int NF, int DIMS, bool PAIRS>
__global__ void __launch_bounds__(kDiagThreads, sizeof(T) == 4 && NF <= 2 ? 4 : 1) k_diag(const DiagArgs<T> p, const DiagTasks tk) {
  constexpr int NV = 4 * NF + 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t N = p.N;
  const DiagScalars<T> k = diag_scalars(p);
  const int raw_u = p.raw_u;
  __shared__ double big[NV];
  if (threadIdx.x < NV) big[threadIdx.x] = 0.0;
  __syncthreads();
  RunningSums<T, NV> acc;
  acc.clear();
  T shift[NF];
#pragma unroll
  for (int i = 0; i < NF; ++i) shift[i] = p.f[i][0];
  if constexpr (DIMS == 1) {
    for (int64_t task = blockIdx.x; task < tk.count; task += gridDim.x) {
      Partials<T, NV, PAIRS> part;
      part.clear();
      const int64_t s0 = task * (kDiagThreads * (sizeof(T) == 8 ? tk.len : kFlush)) + threadIdx.x;
      const int len = sizeof(T) == 8 ? tk.len : kFlush;
#pragma unroll 4
      for (int r = 0; r < len; ++r) {
        const int64_t s = s0 + r * kDiagThreads;
        if (s >= p.S) break;
        T f[NF], w[NF], nb[NF][1][2];
#pragma unroll
        for (int i = 0; i < NF; ++i) {
          f[i] = __ldg(p.f[i] + s);
          w[i] = __ldg(p.w[i] + s);
          nb[i][0][0] = __ldg(p.f[i] + (s == N - 1 ? 0 : s + 1));
          nb[i][0][1] = __ldg(p.f[i] + (s == 0 ? N - 1 : s - 1));
        }
        diag_site<PAIRS, T, NF, 1>(k, raw_u, f, w, nb, shift, part);
      }
      __syncwarp();
      acc.add(part, big);
    }
  } else {
    const int64_t plane = DIMS == 3 ? N * N : N;               // stride of the sweep axis
    for (int64_t task = blockIdx.x; task < tk.count; task += gridDim.x) {
      // the lane's column: (x, y) in 3D, x in 2D; columns past the lattice's end
      // repeat its last one and add nothing
      // FP64: the chunks of a column group follow one another (a plane's last group, which
      // may hold few sites, goes to blocks that have a task already)
      const int64_t inner = sizeof(T) == 8 ? tk.count / tk.nx : tk.nx;
      const int xs = (int)(sizeof(T) == 8 ? task / inner : task % inner);
      const int64_t rest = sizeof(T) == 8 ? task % inner : task / inner;
      const int n = (int)N;                                    // sides below 2^17
      int x, y = 0, chunk;
      bool site;
      if constexpr (DIMS == 3 && sizeof(T) == 8) {
        const int at = xs * kDiagThreads + threadIdx.x;
        site = at < n * n;
        y = min(at, n * n - 1) / n;
        x = min(at, n * n - 1) - y * n;
        chunk = (int)rest;
      } else {
        if constexpr (DIMS == 3) {
          x = xs * 32 + lane;
          y = (int)(rest % tk.ny) * kDiagWarps + warp;
          chunk = (int)(rest / tk.ny);
        } else {
          x = xs * kDiagThreads + threadIdx.x;
          chunk = (int)rest;
        }
        site = x < n && y < n;
        x = min(x, n - 1);
        y = min(y, n - 1);
      }
      // offsets in a plane, added to the plane's (uniform) base
      const uint32_t o = (uint32_t)y * (uint32_t)n + x;
      const uint32_t oxp = x == n - 1 ? o - (n - 1) : o + 1, oxm = x == 0 ? o + (n - 1) : o - 1;
      const uint32_t column = (uint32_t)(n - 1) * (uint32_t)n;   // used in 3D only, where it fits
      const uint32_t oyp = y == n - 1 ? o - column : o + n, oym = y == 0 ? o + column : o - n;
      const int z0 = chunk * tk.len;
      int z1 = min(z0 + tk.len, n);
      if constexpr (sizeof(T) == 8) z1 = __any_sync(0xffffffffu, site) ? z1 : z0;   // no site: nothing to sum
      T fm[NF], fc[NF];
      Partials<T, NV, PAIRS> part;
      part.clear();
#pragma unroll
      for (int i = 0; i < NF; ++i) {
        fm[i] = __ldg(p.f[i] + (z0 == 0 ? n - 1 : z0 - 1) * plane + o);
        fc[i] = __ldg(p.f[i] + z0 * plane + o);
      }
      constexpr int kUnroll = sizeof(T) == 8 ? 1 : (NF <= 2 ? 2 : 4);
#pragma unroll kUnroll
      for (int z = z0; z < z1; ++z) {
        const int64_t here = z * plane, next = (z + 1 == n ? 0 : z + 1) * plane;
        T w[NF], nb[NF][DIMS][2], fn[NF];
#pragma unroll
        for (int i = 0; i < NF; ++i) {
          const T* fz = p.f[i] + here;
          fn[i] = __ldg(p.f[i] + next + o);
          w[i] = __ldg(p.w[i] + here + o);
          nb[i][0][0] = __ldg(fz + oxp);
          nb[i][0][1] = __ldg(fz + oxm);
          if constexpr (DIMS == 3) {
            nb[i][1][0] = __ldg(fz + oyp);
            nb[i][1][1] = __ldg(fz + oym);
          }
          nb[i][DIMS - 1][0] = fn[i];
          nb[i][DIMS - 1][1] = fm[i];
        }
        diag_site<PAIRS, T, NF, DIMS>(k, raw_u, fc, w, nb, shift, part);
#pragma unroll
        for (int i = 0; i < NF; ++i) {
          fm[i] = fc[i];
          fc[i] = fn[i];
        }
      }
      if (!site) part.clear();   // the whole warp takes part in the addition
      __syncwarp();
      acc.add(part, big);
    }
  }
  diag_finish<T, NF, NV>(p, acc, big);
}

// Energies of an expanding FP32 run's starting state (w is u), from which a'(0) and
// a''(0) follow and with them float(c) of every step.  What a thread adds in FP32 is 16
// sites at the grid's stride: any other 16 are as near to the exact sums (1e-8), but
// float(c) would round otherwise now and then, and from then on every site's rounding,
// so a run would end off by its own rounding error (2e-5 of the velocities after 1000
// steps).  No field moments.
template <int NF, int DIMS>
__global__ void __launch_bounds__(kDiagThreads, NF <= 2 ? 4 : 2) k_start_sums(const DiagArgs<float> p) {
  constexpr int NV = 2 * NF + 1;
  __shared__ double big[NV];
  if (threadIdx.x < NV) big[threadIdx.x] = 0.0;
  __syncthreads();
  RunningSums<float, NV> acc;
  acc.clear();
  const int64_t N = p.N, stride = (int64_t)gridDim.x * kDiagThreads;
  const int64_t plane = DIMS == 3 ? N * N : N;
  int64_t s = (int64_t)blockIdx.x * kDiagThreads + threadIdx.x;
  // coordinates of s and of the stride (1D: x is s)
  const int n = DIMS == 1 ? 0 : (int)N;
  int x = 0, y = 0, z = 0, dx = 0, dy = 0, dz = 0;
  if constexpr (DIMS >= 2) {
    x = (int)(s % N);
    dx = (int)(stride % N);
    y = (int)(DIMS == 3 ? s / N % N : s / N);
    dy = (int)(DIMS == 3 ? stride / N % N : stride / N);
  }
  if constexpr (DIMS == 3) {
    z = (int)(s / plane);
    dz = (int)(stride / plane);
  }
  const float q[3] = {(float)p.q[0], (float)p.q[1], (float)p.q[2]};
  const int64_t groups = ((p.S + stride - 1) / stride + kFlush - 1) / kFlush;
  for (int64_t g = 0; g < groups; ++g) {
    Partials<float, NV, false> part;
    part.clear();
#pragma unroll 4
    for (int r = 0; r < kFlush; ++r) {
      if (s >= p.S) break;
      int64_t up[DIMS];   // the neighbours at +e_d
      up[0] = (DIMS == 1 ? s == N - 1 : x == n - 1) ? s - (N - 1) : s + 1;
      if constexpr (DIMS >= 2) up[1] = y == n - 1 ? s - (N - 1) * N : s + N;
      if constexpr (DIMS == 3) up[2] = z == n - 1 ? s - (N - 1) * plane : s + plane;
      float f[NF], dv[NF], vs;
#pragma unroll
      for (int i = 0; i < NF; ++i) {
        f[i] = __ldg(p.f[i] + s);
        const float u = __ldg(p.w[i] + s);
        float g2 = 0.f;
#pragma unroll
        for (int d = 0; d < DIMS; ++d) {
          const float df = __ldg(p.f[i] + up[d]) - f[i];
          g2 = fmaf(df, df, g2);
        }
        part.v[i] = fmaf(0.5f * u, u, part.v[i]);
        part.v[NF + i] += g2;
      }
      model_dv<float, NF>(f, q, dv, vs);
      part.v[2 * NF] += vs;
      s += stride;
      if constexpr (DIMS >= 2) {   // in range again after one subtraction each
        x += dx;
        y += dy;
        if (x >= n) {
          x -= n;
          ++y;
        }
      }
      if constexpr (DIMS == 3) {
        z += dz;
        if (y >= n) {
          y -= n;
          ++z;
        }
      }
    }
    __syncwarp();
    acc.add(part, big);
  }
  diag_finish<float, NF, NV>(p, acc, big);
}

// A grid that is resident as a whole (at most `cap` blocks): tasks are strided.
template <typename T, int NF, int DIMS, bool PAIRS>
cudaError_t launch_diag_kernel(const DiagArgs<T>& a, int cap, cudaStream_t st) {
  int per_sm = 1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_diag<T, NF, DIMS, PAIRS>, kDiagThreads, 0) !=
          cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  cap = std::min(cap, per_sm * sm_count(-1));
  const DiagTasks tk = diag_tasks(DIMS, sizeof(T) == 8, a.N, a.S, cap);
  const int blocks = (int)std::min<int64_t>(tk.count, cap);
  k_diag<T, NF, DIMS, PAIRS><<<blocks, kDiagThreads, 0, st>>>(a, tk);
  return cudaGetLastError();
}

template <typename T, int NF, int DIMS>
cudaError_t launch_diag_dims(const DiagArgs<T>& a, int cap, cudaStream_t st) {
  if constexpr (sizeof(T) == 4) {
    if (a.raw_u && a.expansion) {
      const int blocks = (int)std::min<int64_t>((a.S + kDiagThreads - 1) / kDiagThreads, cap);
      k_start_sums<NF, DIMS><<<blocks, kDiagThreads, 0, st>>>(a);
      return cudaGetLastError();
    }
    if (a.S < kPairSites) return launch_diag_kernel<T, NF, DIMS, true>(a, cap, st);
  }
  return launch_diag_kernel<T, NF, DIMS, false>(a, cap, st);
}

template <typename T, int NF>
cudaError_t launch_diag_nf(const DiagArgs<T>& a, int cap, cudaStream_t st) {
  switch (a.dims) {
    case 1: return launch_diag_dims<T, NF, 1>(a, cap, st);
    case 2: return launch_diag_dims<T, NF, 2>(a, cap, st);
    default: return launch_diag_dims<T, NF, 3>(a, cap, st);
  }
}

}  // namespace

template <typename T>
cudaError_t launch_diag(const DiagArgs<T>& a, int cap, cudaStream_t st) {
  switch (a.nf) {
    case 1: return launch_diag_nf<T, 1>(a, cap, st);
    case 2: return launch_diag_nf<T, 2>(a, cap, st);
    case 3: return launch_diag_nf<T, 3>(a, cap, st);
    default: return launch_diag_nf<T, 4>(a, cap, st);
  }
}
template cudaError_t launch_diag<float>(const DiagArgs<float>&, int, cudaStream_t);
template cudaError_t launch_diag<double>(const DiagArgs<double>&, int, cudaStream_t);

}  // namespace ce
