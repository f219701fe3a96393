// ce_fx64.cu -- the FP64 step for any dimension and side: drift, kick and the
// energy sum in FP64, the force of every site in integer arithmetic (ce_fx.cuh).
//
// Fused step (arXiv:0712.0813 Sec. III staggered leapfrog), per site and field:
//   v = w + c f,  g = f + dt v                       2 FP64 operations
//   force = raw(g) - dx^2 dV/df(g)                   integers
//   w_out = v + (dt / dx^2) force,  f_out = g        1 FP64 operation
//   sum of the energy terms (expansion only)         1 FP64 operation a site
// What bounds it.  GB300 has two FP64 lanes per clock and SM, so the step in FP64
// (a pass for g, a pass for the stencil, 32 operations a site with two fields) ran
// at 0.85 of that pipe and 0.15 of HBM.  Here 10.2 FP64 operations a site remain
// (256^3 by ncu, halo lanes included; half of that pipe) among 835 instructions, most
// of them integer.  616 us a step at 256^3 (two passes: 1058; 596 with 782 instructions
// when the model force was still cut to the unit of the fields): bound by issue and its
// latency, 0.62 of the issue slots with 17 warps an SM (96 registers a thread), beside
// 0.26 of HBM.
//
// Layout.  A warp holds a strip of 30 x-sites, lane l the column x0 - 1 + l, so lanes 0
// and nx + 1 carry the x-halo and x-neighbours come by shuffles.  3D: a block of RB + 2
// warps, one row each, sweeps a chunk of z; rows above and below are read from a ring of
// planes in shared memory, z-neighbours are the lane's own registers.  2D: a warp sweeps
// a chunk of y by itself, y-neighbours in registers.  1D: one strip at a time, no sweep.
// Each plane's values are converted to integers once, when g is formed.  Any side, no
// alignment.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "ce_device.cuh"
#include "ce_fx_force.cuh"
#include "ce_internal.h"
#include "ce_plan.h"
#include "ce_tma.cuh"

namespace ce {
namespace {

using fx::Fx;

constexpr int kFxWarps = 4;
constexpr int kFxThreads = 32 * kFxWarps;
constexpr int kStrip = 30;   // sites a warp updates along x

__device__ __forceinline__ Fx shfl_up(const Fx& x) {
  return Fx{__shfl_up_sync(0xffffffffu, x.m, 1), __shfl_up_sync(0xffffffffu, x.e, 1)};
}
__device__ __forceinline__ Fx shfl_down(const Fx& x) {
  return Fx{__shfl_down_sync(0xffffffffu, x.m, 1), __shfl_down_sync(0xffffffffu, x.e, 1)};
}

// End of a step from the threads' energy terms: 2 G + 3 V = -dx^-2 <energy>.
__device__ __forceinline__ void finish(const StepArgs<double>& p, double energy) {
  finish_step(p, block_sum(energy) * -p.source.wg);
}

// ---- 3D ---------------------------------------------------------------------
// A block owns 30 x-sites by RB rows and sweeps a chunk of z: RB + 2 warps, one
// row each, the first and the last holding the y-halo rows, which only form g.
// Every warp puts its row of the newest plane into shared memory, where the rows
// above and below read it when that plane is the one being updated; x-neighbours
// come by shuffles, z-neighbours are the lane's own registers.  Two mbarriers, for
// the planes of either parity, count the warps that have put their row in; a warp
// waits for a plane only one plane after putting its own row (a block barrier in
// their place held every warp for 1.9 of 8.4 cycles an instruction), and the ring
// of four planes keeps a row until the slowest warp is done with it.  The waits are
// bounded (CE_ETIMEOUT).
template <int NF>
struct FxRows {
  static constexpr int value = 8;
  static constexpr int blocks = NF <= 2 ? 2 : 1;   // resident blocks per SM the registers are bounded for
};

template <int NF, int RB, bool SUMS>
__global__ void __launch_bounds__(32 * (RB + 2), FxRows<NF>::blocks)
    k_step_fx3(const StepArgs<double> p, const fx::FxModel k, int nstrips, int zlen) {
  __shared__ int64_t sm[4][NF][RB + 2][32];
  __shared__ int se[4][NF][RB + 2][32];
  __shared__ __align__(8) uint64_t bar[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    const uint32_t rows = RB + 2 + p.missing_tx;   // one more where a test makes the waits run out
    mbar_init(&bar[0], rows);
    mbar_init(&bar[1], rows);
    fence_mbar_init();
  }
  __syncthreads();
  const int N = (int)p.N;
  const int64_t NN = (int64_t)N * N;
  const int x0 = (int)(blockIdx.x % nstrips) * kStrip, y0 = (int)(blockIdx.x / nstrips) * RB;
  const int nx = min(kStrip, N - x0);
  const int z0 = blockIdx.y * zlen, z1 = min(z0 + zlen, N);
  const int np = z1 - z0 + 2;                    // planes z0 - 1 .. z1
  int xs = x0 - 1 + min(lane, nx + 1);
  xs = xs < 0 ? xs + N : (xs >= N ? xs - N : xs);
  int y = y0 - 1 + warp;                         // rows past the lattice's end wrap and update nothing
  const bool row = warp >= 1 && warp <= RB && y < N;
  y = y < 0 ? y + N : y % N;
  const bool site = row && lane >= 1 && lane <= nx;
  const int64_t here = (int64_t)y * N + xs;
  // the lane's site in the planes under way, formed and updated: z0 - 1 + j (mod N)
  int zq = z0 == 0 ? N - 1 : z0 - 1;
  int64_t oq = zq * NN + here, oN = oq, oC = oq;
  const double c = p.sc_in->c, dd = p.dt_drift, kk = p.dt_kick * p.inv_dx2;
  const double q[3] = {p.q[0], p.q[1], p.q[2]};
  double lf[NF], lw[NF];                         // loads under way: the next plane to form
  const auto issue = [&]() {
    const int64_t o = oq;
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      lf[i] = __ldg(p.f_in[i] + o);
      lw[i] = __ldg(p.w_in[i] + o);
    }
  };
  const auto form = [&](int j, Fx (&g)[NF], double (&v)[NF]) {
    const int buf = (j + 3) & 3;
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      v[i] = fma(c, lf[i], lw[i]);
      const double gd = fma(dd, v[i], lf[i]);
      g[i] = fx::from_double(gd);
      if (site && j >= 1 && j <= np - 2) p.f_out[i][oN] = gd;
      sm[buf][i][warp][lane] = g[i].m;
      se[buf][i][warp][lane] = g[i].e;
    }
    __syncwarp();
    if (lane == 0 && j >= 1) mbar_arrive(&bar[(j - 1) & 1]);
  };
  // every row of plane j is in shared memory
  const auto wait_plane = [&](int j) -> bool {
    uint64_t* b = &bar[(j - 1) & 1];
    const uint32_t parity = (uint32_t)((j - 1) >> 1) & 1u;
    if (mbar_try_wait(b, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(b, parity))
      if (clock64() - t0 > p.wait_cycles) return false;
    return true;
  };
  double acc = 0.0;
  Fx gP[NF], gC[NF], gN[NF];
  double vC[NF], vN[NF];
  const auto advance = [&]() {                   // the plane under way is the next to form
    oC = oN;
    oN = oq;
    if (++zq == N) {
      zq = 0;
      oq = here;
    } else {
      oq += NN;
    }
  };
  issue();
  advance();
  form(0, gP, vC);
  issue();
  advance();
  form(1, gC, vC);
  issue();
#pragma unroll 1
  for (int j = 1; j <= np - 2; ++j) {
    advance();                                   // oC: plane j, oN: plane j + 1, oq: plane j + 2
    form(j + 1, gN, vN);
    if (j + 2 < np) issue();
    if (!__all_sync(0xffffffffu, wait_plane(j))) {
      if (lane == 0) atomicCAS(p.status, CE_OK, CE_ETIMEOUT);
      break;
    }
    if (row) {
      const int cur = (j + 3) & 3;
      Fx nb[NF][6];
#pragma unroll
      for (int i = 0; i < NF; ++i) {
        nb[i][0] = shfl_up(gC[i]);
        nb[i][1] = shfl_down(gC[i]);
        nb[i][2] = Fx{sm[cur][i][warp - 1][lane], se[cur][i][warp - 1][lane]};
        nb[i][3] = Fx{sm[cur][i][warp + 1][lane], se[cur][i][warp + 1][lane]};
        nb[i][4] = gP[i];
        nb[i][5] = gN[i];
      }
      if (site) {
        double force[NF], energy;
        fx::force_of<NF, 3, SUMS>(gC, nb, k, p.inv_dx2, q, force, energy);
        if constexpr (SUMS) acc += energy;
#pragma unroll
        for (int i = 0; i < NF; ++i) p.w_out[i][oC] = fma(kk, force[i], vC[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      gP[i] = gC[i];
      gC[i] = gN[i];
      vC[i] = vN[i];
    }
  }
  __syncthreads();
  if constexpr (SUMS) finish(p, acc);
}

// ---- 2D ---------------------------------------------------------------------
template <int NF, bool SUMS>
__global__ void __launch_bounds__(kFxThreads, 3) k_step_fx2(const StepArgs<double> p, const fx::FxModel k, int nstrips,
                                                          int ylen) {
  constexpr int DL = 2;   // rows of loads under way
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t N = p.N;
  const int64_t wg = (int64_t)blockIdx.x * kFxWarps + warp;
  double acc = 0.0;
  if (wg < nstrips) {
    const int64_t x0 = wg * kStrip;
    const int nx = (int)min((int64_t)kStrip, N - x0);
    int64_t xs = x0 - 1 + min(lane, nx + 1);
    xs = xs < 0 ? xs + N : (xs >= N ? xs - N : xs);
    const bool site = lane >= 1 && lane <= nx;
    const int y0 = blockIdx.y * ylen;
    const int y1 = (int)min((int64_t)y0 + ylen, N);
    const int n = y1 - y0 + 2;                     // rows y0 - 1 .. y1
    const auto row_off = [&](int j) -> int64_t {
      int64_t y = (int64_t)y0 - 1 + j;
      y = y < 0 ? y + N : (y >= N ? y - N : y);
      return y * N + xs;
    };
    const double c = p.sc_in->c, dd = p.dt_drift, kk = p.dt_kick * p.inv_dx2;
    const double q[3] = {p.q[0], p.q[1], p.q[2]};
    double lf[DL][NF], lw[DL][NF];
    const auto issue = [&](int j, int slot) {
      const int64_t o = row_off(j);
#pragma unroll
      for (int i = 0; i < NF; ++i) {
        lf[slot][i] = __ldg(p.f_in[i] + o);
        lw[slot][i] = __ldg(p.w_in[i] + o);
      }
    };
#pragma unroll
    for (int s = 0; s < DL; ++s)
      if (s < n) issue(s, s);
    Fx gm[NF], gc[NF], gp[NF];
    double vc[NF], vp[NF];
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      gm[i] = gc[i] = gp[i] = Fx{0, 1};
      vc[i] = vp[i] = 0.0;
    }
    for (int j0 = 0; j0 < n; j0 += DL) {
#pragma unroll
      for (int s = 0; s < DL; ++s) {
        const int j = j0 + s;
        if (j >= n) break;
        const int64_t oj = row_off(j);
        const bool own = site && j >= 1 && j <= n - 2;
#pragma unroll
        for (int i = 0; i < NF; ++i) {
          const double v = fma(c, lf[s][i], lw[s][i]);
          const double g = fma(dd, v, lf[s][i]);
          gm[i] = gc[i];
          gc[i] = gp[i];
          gp[i] = fx::from_double(g);
          vc[i] = vp[i];
          vp[i] = v;
          if (own) p.f_out[i][oj] = g;
        }
        if (j + DL < n) issue(j + DL, s);
        if (j < 2) continue;
        Fx nb[NF][4];
#pragma unroll
        for (int i = 0; i < NF; ++i) {
          nb[i][0] = shfl_up(gc[i]);
          nb[i][1] = shfl_down(gc[i]);
          nb[i][2] = gm[i];
          nb[i][3] = gp[i];
        }
        if (site) {
          double force[NF], energy;
          fx::force_of<NF, 2, SUMS>(gc, nb, k, p.inv_dx2, q, force, energy);
          if constexpr (SUMS) acc += energy;
          const int64_t o = row_off(j - 1);
#pragma unroll
          for (int i = 0; i < NF; ++i) p.w_out[i][o] = fma(kk, force[i], vc[i]);
        }
      }
    }
  }
  if constexpr (SUMS) finish(p, acc);
}

// ---- 1D ---------------------------------------------------------------------
template <int NF, bool SUMS>
__global__ void __launch_bounds__(kFxThreads) k_step_fx1(const StepArgs<double> p, const fx::FxModel k, int64_t nstrips) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t N = p.N, stride = (int64_t)gridDim.x * kFxWarps;
  const double c = p.sc_in->c, dd = p.dt_drift, kk = p.dt_kick * p.inv_dx2;
  const double q[3] = {p.q[0], p.q[1], p.q[2]};
  double acc = 0.0;
  const auto column = [&](int64_t strip) -> int64_t {
    const int64_t x0 = strip * kStrip, nx = min((int64_t)kStrip, N - x0);
    const int64_t x = x0 - 1 + min((int64_t)lane, nx + 1);
    return x < 0 ? x + N : (x >= N ? x - N : x);
  };
  double lf[NF], lw[NF];
  const auto issue = [&](int64_t strip) {
    const int64_t x = column(strip);
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      lf[i] = __ldg(p.f_in[i] + x);
      lw[i] = __ldg(p.w_in[i] + x);
    }
  };
  int64_t strip = (int64_t)blockIdx.x * kFxWarps + warp;
  if (strip < nstrips) issue(strip);
  for (; strip < nstrips; strip += stride) {
    const int64_t x = column(strip);
    const bool site = lane >= 1 && lane <= min((int64_t)kStrip, N - strip * kStrip);
    Fx g[NF], nb[NF][2];
    double v[NF];
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      v[i] = fma(c, lf[i], lw[i]);
      const double gd = fma(dd, v[i], lf[i]);
      g[i] = fx::from_double(gd);
      if (site) p.f_out[i][x] = gd;
    }
    if (strip + stride < nstrips) issue(strip + stride);
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      nb[i][0] = shfl_up(g[i]);
      nb[i][1] = shfl_down(g[i]);
    }
    if (site) {
      double force[NF], energy;
      fx::force_of<NF, 1, SUMS>(g, nb, k, p.inv_dx2, q, force, energy);
      if constexpr (SUMS) acc += energy;
#pragma unroll
      for (int i = 0; i < NF; ++i) p.w_out[i][x] = fma(kk, force[i], v[i]);
    }
  }
  if constexpr (SUMS) finish(p, acc);
}

// ---- host -------------------------------------------------------------------

// x as a 64-bit fraction in [1/2, 1) and a power of two.
fx::FxConst constant(long double x) {
  fx::FxConst c{0, -4096};
  if (!(x > 0.0L)) return c;
  int e = 0;
  c.m = (uint64_t)std::ldexp(std::frexp(x, &e), 64);
  c.e = e;
  return c;
}

// The kernels kick by kk force with kk = dt / dx^2 rounded to FP64, so the dx^2
// inside the force is dt / kk to 64 bits: the model force then enters with dt
// itself (with both constants rounded to FP64 the potential of the oscillating mean
// field was off by 2e-14 after 1000 steps, 3e-15 with dt).
}  // namespace

fx::FxModel fx_model(double dt_kick, double inv_dx2, const double* q) {
  fx::FxModel k;
  const volatile double kk = dt_kick * inv_dx2;   // the kernels' own product
  const long double dx2 = (long double)dt_kick / (long double)kk;
  k.dx2 = constant(dx2);
  for (int i = 0; i < 3; ++i) {
    k.q[i] = constant(q[i]);
    k.qdx2[i] = constant((long double)q[i] * dx2);
  }
  return k;
}

namespace {

template <int NF, bool SUMS>
const void* kernel_of(int dims) {
  return dims == 3 ? (const void*)k_step_fx3<NF, FxRows<NF>::value, SUMS>
                   : (dims == 2 ? (const void*)k_step_fx2<NF, SUMS> : (const void*)k_step_fx1<NF, SUMS>);
}
template <int NF>
const void* kernel_nf(int dims, bool sums) {
  return sums ? kernel_of<NF, true>(dims) : kernel_of<NF, false>(dims);
}
const void* kernel(int dims, int nf, bool sums) {
  switch (nf) {
    case 1: return kernel_nf<1>(dims, sums);
    case 2: return kernel_nf<2>(dims, sums);
    case 3: return kernel_nf<3>(dims, sums);
    default: return kernel_nf<4>(dims, sums);
  }
}

template <int NF, bool SUMS>
void launch(const StepArgs<double>& a, const FxPlan& pl, cudaStream_t st) {
  const fx::FxModel k = fx_model(a.dt_kick, a.inv_dx2, a.q);
  const dim3 grid(pl.gx, pl.gy);
  if (a.dims == 3)
    k_step_fx3<NF, FxRows<NF>::value, SUMS><<<grid, 32 * (FxRows<NF>::value + 2), 0, st>>>(a, k, pl.nstrips, pl.len);
  else if (a.dims == 2) k_step_fx2<NF, SUMS><<<grid, kFxThreads, 0, st>>>(a, k, pl.nstrips, pl.len);
  else k_step_fx1<NF, SUMS><<<grid, kFxThreads, 0, st>>>(a, k, (a.N + kStrip - 1) / kStrip);
}
template <int NF>
void launch_nf(const StepArgs<double>& a, const FxPlan& pl, cudaStream_t st) {
  if (a.update_scalars) launch<NF, true>(a, pl, st);
  else launch<NF, false>(a, pl, st);
}

}  // namespace

// Strips and row groups as in the column and line-sweep kernels; the chunk along
// the sweep from the wave model (ce_plan.h), a chunk paying about 3 planes for
// its two halo planes and its start.
FxPlan fx_plan(int dims, int64_t N, int nf, int sms) {
  FxPlan pl{};
  const int rows = nf <= 2 ? FxRows<2>::value : FxRows<4>::value;
  const int threads = dims == 3 ? 32 * (rows + 2) : kFxThreads;
  int per_sm = 1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel(dims, nf, true), threads, 0) != cudaSuccess) {
    cudaGetLastError();
    per_sm = 1;
  }
  const int64_t slots = (int64_t)std::max(per_sm, 1) * sms;
  const int64_t strips = (N + kStrip - 1) / kStrip;
  pl.gy = 1;
  if (dims == 1) {
    pl.nstrips = 0;   // more than an int holds on the longest lines: formed from N
    pl.gx = (int)std::min<int64_t>((strips + kFxWarps - 1) / kFxWarps, slots);
    return pl;
  }
  pl.nstrips = (int)strips;
  pl.gx = (int)(dims == 3 ? strips * ((N + rows - 1) / rows) : (strips + kFxWarps - 1) / kFxWarps);
  pl.len = plan::wave_chunk_length(N, pl.gx, slots, 1, 3.0);
  pl.gy = (int)((N + pl.len - 1) / pl.len);
  return pl;
}

cudaError_t launch_step_fx(const StepArgs<double>& a, const FxPlan& pl, cudaStream_t st) {
  switch (a.nf) {
    case 1: launch_nf<1>(a, pl, st); break;
    case 2: launch_nf<2>(a, pl, st); break;
    case 3: launch_nf<3>(a, pl, st); break;
    default: launch_nf<4>(a, pl, st); break;
  }
  return cudaGetLastError();
}

}  // namespace ce
