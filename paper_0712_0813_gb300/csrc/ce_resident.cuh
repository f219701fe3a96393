// ce_resident.cuh -- many steps of a small lattice in one cooperative launch.
//
// A lattice of some 10^5 sites takes a few microseconds a step whatever its
// kernel: a launch, the first loads, the block sums, and the last block's tail (sum
// of the partials, a', the end of the grid) follow one another.  Here the lattice
// stays in the shared memory of at most one block per SM for the steps of a ce_step call.
// Each block owns a brick of the lattice; per step it
//   1. waits until every block has published the last step (a counter),
//   2. loads f and w of its halo from L2, while one warp sums the blocks' shares of
//      2 G + 3 V and advances a, a', a'' (every block the same way),
//   3. forms g = f + dt (w + c f) of its sites and its halo in shared memory,
//   4. updates its sites from there, stores the brick's surface for the neighbours
//      (all of it in the last step) and publishes its share.
// One grid-wide exchange a step.  Shares and surfaces alternate between two buffers:
// a block writes one again only after every block has published the step after it.
// Waits are bounded (CE_ETIMEOUT); the cooperative launch keeps all blocks resident.
//
// What bounds a step is latency: the exchange 2430 cycles between 152 blocks (release,
// counter, acquire; 6500 when every block polled every other's tagged entry, whose
// lines then serve 152 readers), the halo and the shares, the FP64 chain of a'.
#pragma once

#include <algorithm>
#include <cstdint>

#include "ce_device.cuh"
#include "ce_fx_force.cuh"
#include "ce_internal.h"

namespace ce {
namespace resident {

// Most threads of a block, and resident blocks per SM the registers are bounded for.
// FP64 with three and four fields spilt at 512 threads (four at 33^3: 13.3 us a step,
// 11.9 at 384, two dimensions at 400^2 16.9 and 15.6).
template <typename T, int NF>
struct Shape {
  static constexpr int threads = sizeof(T) == 8 && NF > 2 ? 384 : 512;
  static constexpr int blocks = sizeof(T) == 8 ? 1 : 2;
};

// Blocks and threads.  A block per SM and a thread per site would be the shortest step
// of a lattice that has the GPU to itself, but not by much: half the SMs serve small
// lattices as well (fewer blocks in the exchange), and two to four sites a thread hide
// their own latency.  What is left free lets other handles' launches run beside this
// one.  us a step, two fields, expanding, one handle / 16 handles on their own streams,
// with a thread per site on every SM and as below: FP32 20^3 4.2 / 0.75 and 3.9 / 0.52,
// 32^3 4.3 / 1.55 and 4.8 / 0.83, 48^3 5.6 / 5.6 and 5.4 / 2.0, 64^3 7.4 / 7.3 and
// 7.0 / 4.6; 2D 300^2 4.9 / 4.9 and 4.9 / 1.5, 700^2 7.7 / 7.6 and 7.2 / 4.4; FP64 16^3
// 5.5 / 1.4 and 5.5 / 0.76, 48^3 10.2 / 10.2 and 10.1 / 6.9, 1D 65536 7.3 / 7.3 and
// 7.1 / 4.1.
template <typename T>
int blocks_limit(int64_t S, int sms) {
  return S <= (sizeof(T) == 4 ? 70000 : 12000) ? std::max(1, sms / 2) : sms;
}
template <typename T>
int threads_limit(int dims, int nf, int64_t sites, int64_t halo) {
  if (sizeof(T) == 4) return sites + halo <= (dims == 3 ? 1500 : 2500) ? 256 : 512;
  return sites * nf <= 2000 ? 256 : (nf > 2 ? Shape<T, 4>::threads : Shape<T, 2>::threads);
}

constexpr size_t kStaticSmem = 8192;   // room left for the kernel's static shared memory
constexpr int kHeld = 2;   // halo sites a thread holds in registers while a' is formed

// Consecutive sites of which a thread adds the energy terms in T before they join its
// running sums: four in 1D and FP32, one else.  These are the sums of the kernels that
// take one launch a step (the 1D kernel's 16-byte groups, the generic kernel's sites),
// so a run's a(t), and with it FP32's rounding of every site, does not depend on which
// of them it takes.
template <typename T>
__host__ __device__ constexpr int group(int dims) {
  return dims == 1 && sizeof(T) == 4 ? 4 : 1;
}

// Shared memory of a brick: the tile (g of the padded brick), the velocities of its
// sites, and where each site and halo site lies in the tile and in the lattice.
template <typename T>
__host__ __device__ inline size_t tile_bytes(int nf, int padded) {
  const size_t n = (size_t)nf * padded * (sizeof(T) == 4 ? 4 : 12);
  return (n + 15) / 16 * 16;
}
template <typename T>
__host__ __device__ inline size_t smem_bytes(int nf, int padded, int sites, int halo) {
  return tile_bytes<T>(nf, padded) + ((size_t)nf * sites * sizeof(T) + 15) / 16 * 16 + 6 * (size_t)(sites + halo) + 32;
}

// Halo entry: index of the site in the lattice and place in the padded brick.
struct HaloRef {
  int src, dst;
};

// Brick of block b and its padded layout.
struct Brick {
  int x0, y0, z0, ex, ey, ez;   // origin and extent (shorter at the lattice's end)
  int px, pxy;                  // padded row and plane strides
};

__device__ __forceinline__ Brick brick_of(const ResidentPlan& pl, int N, int dims, int b) {
  Brick k;
  const int ix = b % pl.nx, iy = (b / pl.nx) % pl.ny, iz = b / (pl.nx * pl.ny);
  k.x0 = ix * pl.bx;
  k.y0 = iy * pl.by;
  k.z0 = iz * pl.bz;
  k.ex = min(pl.bx, N - k.x0);
  k.ey = dims >= 2 ? min(pl.by, N - k.y0) : 1;
  k.ez = dims == 3 ? min(pl.bz, N - k.z0) : 1;
  k.px = k.ex + 2;
  k.pxy = dims >= 2 ? k.px * (k.ey + 2) : k.px;
  return k;
}

__device__ __forceinline__ int wrap(int v, int N) { return v < 0 ? v + N : (v >= N ? v - N : v); }

// The h-th halo site: the two x-faces, then the y-faces, then the z-faces.
template <int DIMS>
__device__ __forceinline__ HaloRef halo_ref(const Brick& k, int N, int h) {
  int x, y = 0, z = 0;   // inside the padded brick, interior from 0
  const int fx = k.ey * k.ez, fy = k.ex * k.ez, fz = k.ex * k.ey;
  if (h < 2 * fx) {
    const int side = h >= fx, r = h - side * fx;
    x = side ? k.ex : -1;
    y = r % k.ey;
    z = r / k.ey;
  } else if (DIMS >= 2 && h < 2 * (fx + fy)) {
    h -= 2 * fx;
    const int side = h >= fy, r = h - side * fy;
    y = side ? k.ey : -1;
    x = r % k.ex;
    z = r / k.ex;
  } else {
    h -= 2 * (fx + fy);
    const int side = h >= fz, r = h - side * fz;
    z = side ? k.ez : -1;
    x = r % k.ex;
    y = r / k.ex;
  }
  HaloRef o;
  const int gx = wrap(k.x0 + x, N), gy = DIMS >= 2 ? wrap(k.y0 + y, N) : 0, gz = DIMS == 3 ? wrap(k.z0 + z, N) : 0;
  o.src = (gz * N + gy) * N + gx;
  o.dst = (x + 1) + (DIMS >= 2 ? (y + 1) * k.px : 0) + (DIMS == 3 ? (z + 1) * k.pxy : 0);
  return o;
}

template <int DIMS>
__device__ __forceinline__ int halo_count(const Brick& k) {
  int h = 2 * k.ey * k.ez;
  if (DIMS >= 2) h += 2 * k.ex * k.ez;
  if (DIMS == 3) h += 2 * k.ex * k.ey;
  return h;
}

// g of the padded brick in shared memory: one array per field (FP64: significands
// and exponents in two).
template <typename T>
struct Tile;
template <>
struct Tile<float> {
  float* v;
  int n;   // padded sites
  __device__ __forceinline__ void put(int i, int at, float g) { v[i * n + at] = g; }
  __device__ __forceinline__ float get(int i, int at) const { return v[i * n + at]; }
  __device__ __forceinline__ float value(int i, int at) const { return v[i * n + at]; }
};
template <>
struct Tile<double> {
  int64_t* m;
  int* e;
  int n;
  __device__ __forceinline__ void put(int i, int at, double g) {
    const fx::Fx x = fx::from_double(g);
    m[i * n + at] = x.m;
    e[i * n + at] = x.e;
  }
  __device__ __forceinline__ fx::Fx get(int i, int at) const { return fx::Fx{m[i * n + at], e[i * n + at]}; }
  __device__ __forceinline__ double value(int i, int at) const { return fx::to_double(get(i, at)); }
};

// One site's kick from the tile: w = v + dt F (in w), and its terms of the sums.
template <int NF, int DIMS, bool SUMS>
__device__ __forceinline__ void kick(const ResidentArgs<float>& p, const Tile<float>& t, int at, const int (&st)[3],
                                     float (&w)[NF], float& s0, float& s1) {
  float g[NF], lap[NF], dv[NF], vs;
#pragma unroll
  for (int i = 0; i < NF; ++i) {   // the generic kernel's operations, in its order
    g[i] = t.get(i, at);
    float acc = 0.f;
#pragma unroll
    for (int d = 0; d < DIMS; ++d) {
      const float gp = t.get(i, at + st[d]), gm = t.get(i, at - st[d]);
      acc += (gp + gm) - 2.f * g[i];
      const float df = gp - g[i];
      if (SUMS) s0 = fmaf(df, df, s0);
    }
    lap[i] = acc * p.inv_dx2;
  }
  const float q[3] = {p.q[0], p.q[1], p.q[2]};
  model_dv<float, NF>(g, q, dv, vs);
  if (SUMS) s1 += vs;
#pragma unroll
  for (int i = 0; i < NF; ++i) w[i] = fmaf(p.dt, lap[i] - dv[i], w[i]);
}

template <int NF, int DIMS, bool SUMS>
__device__ __forceinline__ void kick(const ResidentArgs<double>& p, const Tile<double>& t, int at, const int (&st)[3],
                                     double (&w)[NF], double& s0, double&) {
  fx::Fx g[NF], nb[NF][2 * DIMS];
#pragma unroll
  for (int i = 0; i < NF; ++i) {
    g[i] = t.get(i, at);
#pragma unroll
    for (int d = 0; d < DIMS; ++d) {
      nb[i][2 * d] = t.get(i, at + st[d]);
      nb[i][2 * d + 1] = t.get(i, at - st[d]);
    }
  }
  double force[NF], energy;
  const double q[3] = {p.q[0], p.q[1], p.q[2]};
  fx::force_of<NF, DIMS, SUMS, (NF > 3)>(g, nb, p.model, p.inv_dx2, q, force, energy);
  if (SUMS) s0 -= energy;
  const double kk = p.dt * p.inv_dx2;
#pragma unroll
  for (int i = 0; i < NF; ++i) w[i] = fma(kk, force[i], w[i]);
}

// One more block has published its step.
__device__ __forceinline__ void arrive(unsigned* counter) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
}

// Wait until the counter has reached `want` (modulo 2^32); false if that takes too long.
__device__ __forceinline__ bool wait_for(unsigned* counter, unsigned want, long long limit) {
  const long long t0 = clock64();
  for (;;) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
    if ((int)(v - want) >= 0) return true;
    if (clock64() - t0 > limit) return false;
  }
}

template <typename T, int NF, int DIMS, bool SUMS>
__global__ void __launch_bounds__(Shape<T, NF>::threads, Shape<T, NF>::blocks) k_resident(const ResidentArgs<T> p) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ DevScalars s_sc;
  __shared__ int s_abort;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x, nwarps = nthr >> 5;
  const int N = p.N, blocks = gridDim.x;
  const Brick bk = brick_of(p.plan, N, DIMS, blockIdx.x);
  const int sites = bk.ex * bk.ey * bk.ez, halo = halo_count<DIMS>(bk);
  const int padded = DIMS == 1 ? bk.px : (DIMS == 2 ? bk.pxy : bk.pxy * (bk.ez + 2));
  unsigned char* at_mem = smem + tile_bytes<T>(NF, padded);
  T* ws = reinterpret_cast<T*>(at_mem);                               // velocities, [field][site]
  at_mem += ((size_t)NF * sites * sizeof(T) + 15) / 16 * 16;
  int* site_gi = reinterpret_cast<int*>(at_mem);                      // lattice index; sign bit: on the surface
  int* halo_src = site_gi + sites;
  uint16_t* site_at = reinterpret_cast<uint16_t*>(halo_src + halo);   // place in the tile
  uint16_t* halo_at = site_at + sites;
  Tile<T> tile;
  tile.n = padded;
  if constexpr (sizeof(T) == 4) {
    tile.v = reinterpret_cast<float*>(smem);
  } else {
    tile.m = reinterpret_cast<int64_t*>(smem);
    tile.e = reinterpret_cast<int*>(tile.m + (size_t)NF * padded);
  }
  const int st[3] = {1, bk.px, bk.pxy};
  constexpr int G = group<T>(DIMS);

  for (int s = tid; s < sites; s += nthr) {
    const int x = s % bk.ex, y = (s / bk.ex) % bk.ey, z = s / (bk.ex * bk.ey);
    const bool face = x == 0 || x == bk.ex - 1 || (DIMS >= 2 && (y == 0 || y == bk.ey - 1)) ||
                      (DIMS == 3 && (z == 0 || z == bk.ez - 1));
    const int gi = ((bk.z0 + z) * N + bk.y0 + y) * N + bk.x0 + x;
    const int at = (x + 1) + (DIMS >= 2 ? (y + 1) * bk.px : 0) + (DIMS == 3 ? (z + 1) * bk.pxy : 0);
    site_gi[s] = face ? gi | INT32_MIN : gi;
    site_at[s] = (uint16_t)at;
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      tile.put(i, at, p.f[p.in][i][gi]);
      ws[i * sites + s] = p.w[p.in][i][gi];
    }
  }
  for (int h = tid; h < halo; h += nthr) {
    const HaloRef r = halo_ref<DIMS>(bk, N, h);
    halo_src[h] = r.src;
    halo_at[h] = (uint16_t)r.dst;
  }
  if (tid == 0) {
    s_sc = p.slot[p.in];
    s_abort = 0;
  }
  __syncthreads();

  // Thread 0 waits until every block has published step `step`.
  const auto exchange = [&](int step) {
    if (tid == 0 && !wait_for(p.counter, p.count0 + (unsigned)(step + 1) * (unsigned)blocks, p.wait_cycles)) s_abort = 1;
    __syncthreads();
  };
  // Warp 0: the sum of the blocks' shares of a step, and a, a', a'' from it.
  ScaleAhead ahead;
  const auto advance_scalars = [&](int step) {
    const double* shares = p.shares + (size_t)(step & 1) * blocks;
    double sum = 0.0;
    for (int b = lane; b < blocks; b += 32) sum += __ldcg(shares + b);
    sum = warp_sum(sum);
    if (lane == 0) {
      DevScalars out;
      scale_factor_update(ahead, out, sum, p.inv_ddt, p.status);
      s_sc = out;
    }
  };

  int in = p.in;
  for (int step = 0; step < p.steps; ++step) {
    if (step > 0) {
      exchange(step - 1);
      if (s_abort) break;
    }
    // the halo's f and w, on their way while warp 0 advances a'
    T hf[kHeld][NF], hw[kHeld][NF];
#pragma unroll
    for (int j = 0; j < kHeld; ++j) {
      const int h = tid + j * nthr;
      const int src = h < halo ? halo_src[h] : 0;
#pragma unroll
      for (int i = 0; i < NF; ++i) {
        hf[j][i] = h < halo ? __ldcg(p.f[in][i] + src) : T(0);
        hw[j][i] = h < halo ? __ldcg(p.w[in][i] + src) : T(0);
      }
    }
    if (SUMS && step > 0) {
      if (warp == 0) advance_scalars(step - 1);
      __syncthreads();
    }
    const T c = (T)s_sc.c;
    for (int s = tid; s < sites; s += nthr) {   // v = w + c f, g = f + dt v
      const int at = site_at[s];
#pragma unroll
      for (int i = 0; i < NF; ++i) {
        const T f = tile.value(i, at), v = fmaT(c, f, ws[i * sites + s]);
        ws[i * sites + s] = v;
        tile.put(i, at, fmaT(p.dt, v, f));
      }
    }
#pragma unroll
    for (int j = 0; j < kHeld; ++j) {
      const int h = tid + j * nthr;
      if (h < halo) {
        const int at = halo_at[h];
#pragma unroll
        for (int i = 0; i < NF; ++i) tile.put(i, at, fmaT(p.dt, fmaT(c, hf[j][i], hw[j][i]), hf[j][i]));
      }
    }
    for (int h = tid + kHeld * nthr; h < halo; h += nthr) {
#pragma unroll
      for (int i = 0; i < NF; ++i) {
        const T a = __ldcg(p.f[in][i] + halo_src[h]), b = __ldcg(p.w[in][i] + halo_src[h]);
        tile.put(i, halo_at[h], fmaT(p.dt, fmaT(c, a, b), a));
      }
    }
    __syncthreads();
    // kicks; the surface (in the last step every site) to the other buffer
    const bool last = step == p.steps - 1;
    T g0 = T(0), g1 = T(0), v0 = T(0), v1 = T(0);   // the thread's sums (FP32: pairs)
    for (int base = tid * G; base < sites; base += nthr * G) {
      T s0 = T(0), s1 = T(0);
#pragma unroll
      for (int r = 0; r < G; ++r) {
        const int s = base + r;
        if (G > 1 && s >= sites) break;
        const int at = site_at[s], gi = site_gi[s];
        T w[NF];
#pragma unroll
        for (int i = 0; i < NF; ++i) w[i] = ws[i * sites + s];
        kick<NF, DIMS, SUMS>(p, tile, at, st, w, s0, s1);
#pragma unroll
        for (int i = 0; i < NF; ++i) ws[i * sites + s] = w[i];
        if (last || gi < 0) {
          const int o = gi & INT32_MAX;
#pragma unroll
          for (int i = 0; i < NF; ++i) {
            __stcg(p.f[in ^ 1][i] + o, tile.value(i, at));
            __stcg(p.w[in ^ 1][i] + o, w[i]);
          }
        }
      }
      if constexpr (SUMS && sizeof(T) == 4) {
        add_to(g0, g1, s0);
        add_to(v0, v1, s1);
      } else if constexpr (SUMS) {
        g0 += s0;
      }
    }
    in ^= 1;
    // the block's share of 2 G + 3 V; the barriers inside (or the one here) come
    // after every store of the block and every read of the tile
    double share = 0.0;
    if constexpr (!SUMS) __syncthreads();
    else if constexpr (sizeof(T) == 4) share = block_source(g0, g1, v0, v1, p.source);
    else share = block_sum(g0) * p.source.wg;
    if (tid == 0) {
      if (SUMS) __stcg(p.shares + (size_t)(step & 1) * blocks + blockIdx.x, share);
      arrive(p.counter);   // releases the block's stores, ordered before by the barrier
      if (SUMS) ahead = scale_ahead(s_sc, p.ddt, p.kappa2);
    }
  }
  if (SUMS && !s_abort && blockIdx.x == 0) {   // a, a', a'' after the last step
    exchange(p.steps - 1);
    if (warp == 0 && !s_abort) {
      advance_scalars(p.steps - 1);
      if (lane == 0) p.slot[in] = s_sc;
    }
  }
  if (tid == 0 && s_abort) atomicCAS(p.status, CE_OK, CE_ETIMEOUT);
}

// Null where no lattice takes it (plan::resident_takes).
template <typename T, int NF, int DIMS>
const void* kernel_of(bool sums) {
  if (sums) return (const void*)k_resident<T, NF, DIMS, true>;
  if constexpr (sizeof(T) == 8 || DIMS >= 2) return (const void*)k_resident<T, NF, DIMS, false>;
  return nullptr;
}
template <typename T, int NF>
const void* kernel_dims(int dims, bool sums) {
  return dims == 3 ? kernel_of<T, NF, 3>(sums) : (dims == 2 ? kernel_of<T, NF, 2>(sums) : kernel_of<T, NF, 1>(sums));
}
template <typename T>
const void* kernel(int nf, int dims, bool sums) {
  switch (nf) {
    case 1: return kernel_dims<T, 1>(dims, sums);
    case 2: return kernel_dims<T, 2>(dims, sums);
    case 3: return kernel_dims<T, 3>(dims, sums);
    default: return kernel_dims<T, 4>(dims, sums);
  }
}

// The bricks of a lattice: counts per axis with at most one block per SM, the
// least sites plus halo in the largest brick; none where a brick does not fit the
// shared memory.
template <typename T>
ResidentPlan plan(int dims, int64_t N, int nf, int device, int sms) {
  ResidentPlan pl{};
  int64_t S = 1;
  for (int d = 0; d < dims; ++d) S *= N;
  sms = blocks_limit<T>(S, sms);
  int coop = 0, limit = 0;
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, device) != cudaSuccess || !coop ||
      cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess) {
    cudaGetLastError();
    return pl;
  }
  const int n = (int)N;
  const size_t room = (size_t)limit - kStaticSmem;
  int64_t best = INT64_MAX;
  for (int nz = 1; nz <= (dims == 3 ? std::min(n, sms) : 1); ++nz)
    for (int ny = 1; ny <= (dims >= 2 ? std::min(n, sms / nz) : 1); ++ny)
      for (int nx = 1; nx <= std::min(n, sms / (nz * ny)); ++nx) {
        const int g = group<T>(dims), bx = ((n + nx - 1) / nx + g - 1) / g * g, by = dims >= 2 ? (n + ny - 1) / ny : 1, bz = dims == 3 ? (n + nz - 1) / nz : 1;
        // only counts whose last brick is not empty
        if ((nx - 1) * bx >= n || (dims >= 2 && (ny - 1) * by >= n) || (dims == 3 && (nz - 1) * bz >= n)) continue;
        const int64_t sites = (int64_t)bx * by * bz;
        const int64_t halo = 2 * ((int64_t)by * bz + (dims >= 2 ? (int64_t)bx * bz : 0) + (dims == 3 ? (int64_t)bx * by : 0));
        const int64_t padded = (int64_t)(bx + 2) * (dims >= 2 ? by + 2 : 1) * (dims == 3 ? bz + 2 : 1);
        if (padded > 65535) continue;
        const size_t bytes = smem_bytes<T>(nf, (int)padded, (int)sites, (int)halo);
        if (bytes > room) continue;
        if (sites + halo < best) {
          best = sites + halo;
          pl = ResidentPlan{bx, by, bz, nx, ny, nz, nx * ny * nz, 0, (int)bytes};
          const int per = (int)std::min<int64_t>((sites / g + 31) / 32 * 32, threads_limit<T>(dims, nf, sites, halo));
          pl.threads = std::max(per, 128);
        }
      }
  if (pl.blocks == 0) return pl;
  for (int sums = 0; sums < 2; ++sums) {
    const void* k = kernel<T>(nf, dims, sums != 0);
    if (!k) continue;
    int per_sm = 0;
    // one value for every lattice: the attribute is the kernel's, not the handle's
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, pl.threads, pl.smem) != cudaSuccess || per_sm < 1) {
      cudaGetLastError();
      return ResidentPlan{};
    }
  }
  return pl;
}

template <typename T>
cudaError_t launch(const ResidentArgs<T>& a, int dims, int nf, cudaStream_t st) {
  ResidentArgs<T> args = a;
  void* params[] = {&args};
  return cudaLaunchCooperativeKernel(kernel<T>(nf, dims, a.update_scalars != 0), dim3(a.plan.blocks),
                                     dim3(a.plan.threads), params, (size_t)a.plan.smem, st);
}

}  // namespace resident
}  // namespace ce
