// ce_outputs.cu -- outputs beyond the means and energies: the binned power
// spectrum of a field (cuFFT transform + binning kernel), the grid-image file
// (a complete state that ce_load restores exactly; arXiv:0712.0813 Sec. II
// describes grid images that let a run be resumed later), and the state at
// chosen sites (a gather, for probing lattices too large to download).
#include <cuda_runtime.h>
#include <cufft.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "ce_device.cuh"
#include "ce_internal.h"
#include "clusterlat.h"

namespace {

int ofail(int code, const std::string& msg) {
  ce::set_last_error(msg);
  return code;
}

int ocuda(cudaError_t e, const char* what) {
  ce::set_last_error(std::string(what) + ": " + cudaGetErrorString(e));
  return CE_ECUDA;
}

// f(t) and f'(t + dt/2) = w + c f at m chosen sites, for every field; the
// velocity is rounded in T exactly as the step kernels and ce_get_fields form it.
template <typename T>
struct SamplePtrs {
  const T* f[4];
  const T* w[4];
};

template <typename T>
__global__ void k_sample(SamplePtrs<T> p, int nf, const ce::DevScalars* sc, const int64_t* __restrict__ sites,
                         int64_t m, double* __restrict__ out_f, double* __restrict__ out_v) {
  const T c = (T)sc->c;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < m; k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t x = sites[k];
    for (int i = 0; i < nf; ++i) {
      const T fv = p.f[i][x], wv = p.w[i][x];
      out_f[(int64_t)i * m + k] = (double)fv;
      out_v[(int64_t)i * m + k] = (double)ce::fmaT(c, fv, wv);
    }
  }
}

constexpr int kBinThreads = 256;
constexpr int kBinChunks = 16;      // most blocks a bin is shared out to (k_bin_spectrum)
constexpr int kBinParts = 608;      // most partial histograms
constexpr int kRowsSmem = 200 * 1024;   // shared memory of k_bin_rows per SM

// Half-spectrum layout of a real-to-complex transform: the last (x) axis holds
// N/2 + 1 modes.  Every stored mode except kx = 0 and the Nyquist kx = N/2
// stands for itself and its complex conjugate at -n, so it counts twice.
// The transform is taken of f - f(site 0), which keeps the large mean of phi
// out of the FFT's rounding; the zero mode gets S f(site 0) back in FP64.
template <typename T>
__global__ void k_shifted_copy(const T* __restrict__ f, T* __restrict__ out, int64_t n) {
  const T shift = f[0];
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    out[k] = f[k] - shift;
}

// floor(sqrt(x)) for 0 <= x < 2^62: the float root is within 2^-23 of it, which the loops
// make good (no step or one below x = 2^46; lattices end at sides of 2^34 in 1D, where a
// bin's squares reach 2^62).
__device__ __forceinline__ int isqrt(int64_t x) {
  int s = (int)sqrtf((float)x);
  while ((int64_t)s * s > x) --s;
  while ((int64_t)(s + 1) * (s + 1) <= x) ++s;
  return s;
}

// The same for 0 <= x < 2^24, exact in a float.
__device__ __forceinline__ int isqrt(int x) {
  int s;
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"((float)x));   // within one of the root
  s = (int)r;
  s -= s * s > x;
  s += (s + 1) * (s + 1) <= x;
  return s;
}

// w |F|^2 added to a thread's sum: FP64, or for FP32 spectra float pairs (48 bits,
// the squares with their FMA residuals); values whose squares would leave FP32's
// range, infinities and NaN take FP64.
struct PowerSum {
  double wide = 0.0;
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(double re, double im, double w) { wide += w * (re * re + im * im); }
  __device__ __forceinline__ void add(float re, float im, float w) {
    const float big = fmaxf(fabsf(re), fabsf(im)), small = fminf(fabsf(re), fabsf(im));
    if (big < 0x1p50f && (small >= 0x1p-50f || small == 0.f) && (big >= 0x1p-50f || big == 0.f)) {
      const float p = re * re, q = im * im;
      ce::add_to(hi, lo, w * p);
      ce::add_to(hi, lo, w * q);
      lo += w * (fmaf(re, re, -p) + fmaf(im, im, -q));
    } else {
      add((double)re, (double)im, (double)w);
    }
  }
  __device__ __forceinline__ double total() const { return wide + ((double)hi + (double)lo); }
};

// One bin (blockIdx.x) of the spectrum over a share (blockIdx.y) of the rows along x.
// A mode n is in bin b when floor(|n| + 1/2) = b, for integers b^2 - b < n^2 <= b^2 + b
// (bin 0: n = 0), so of the row at (ny, nz) it holds one run of nx, found from two
// square roots.  Threads take rows, so no bin is shared between threads and nothing is
// added atomically (a histogram in shared memory, with a 64-bit division chain, an FP64
// square root and two FP64 compare-and-swap loops a mode, took most of 760 us at 256^3).
// Bounded by the sectors a run touches (L2).
// I: int where every n^2 is below 2^24, else int64_t.
template <typename C, typename T, typename I>
__global__ void __launch_bounds__(kBinThreads) k_bin_spectrum(const C* __restrict__ F, const T* __restrict__ f,
                                                               int64_t N64, int dims, int nbins,
                                                               double* __restrict__ part_p,
                                                               double* __restrict__ part_n) {
  __shared__ double sp[kBinThreads / 32];
  __shared__ unsigned long long sn[kBinThreads / 32];
  const I N = (I)N64, half = N / 2, b = (I)blockIdx.x;
  const int64_t nx = half + 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const I first = b == 0 ? 0 : b * b - b + 1, last = b * b + b;   // n^2 in the bin
  const I kmin = -min(b, (N - 1) / 2), kmax = min(b, half);       // ny, nz that can be in it
  const I zmin = dims == 3 ? kmin : 0, zmax = dims == 3 ? kmax : 0;
  const I ymin = dims >= 2 ? kmin : 0, ymax = dims >= 2 ? kmax : 0;
  // 3D: warps take nz, lanes ny; else every thread takes rows ny
  const I z_at = dims == 3 ? (I)blockIdx.y * (kBinThreads / 32) + warp : 0;
  const I z_by = dims == 3 ? (I)gridDim.y * (kBinThreads / 32) : 1;
  const I y_at = dims == 3 ? (I)lane : (I)blockIdx.y * kBinThreads + threadIdx.x;
  const I y_by = dims == 3 ? 32 : (I)gridDim.y * kBinThreads;
  const double sites = (double)N * (dims >= 2 ? (double)N : 1.0) * (dims == 3 ? (double)N : 1.0);
  PowerSum sum;
  unsigned long long count = 0;
  for (I nz = zmin + z_at; nz <= zmax; nz += z_by)
    for (I ny = ymin + y_at; ny <= ymax; ny += y_by) {
      const I r2 = ny * ny + nz * nz;
      if (r2 > last) continue;
      const int hi = (int)min((I)isqrt(last - r2), half);
      const I from = first - r2;
      const int lo = from <= 0 ? 0 : isqrt(from - 1) + 1;         // ceil(sqrt(from))
      const C* row = F + ((int64_t)(nz < 0 ? nz + N : nz) * N + (ny < 0 ? ny + N : ny)) * nx;
      for (int ix = lo; ix <= hi; ++ix) {
        const bool once = ix == 0 || (N % 2 == 0 && ix == half);
        const C v = row[ix];
        if (b == 0) sum.add((double)v.x + (double)f[0] * sites, (double)v.y, 1.0);   // S f(site 0)
        else sum.add(v.x, v.y, (decltype(v.x))(once ? 1 : 2));
        count += once ? 1 : 2;
      }
    }
  double p = sum.total();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    p += __shfl_down_sync(0xffffffffu, p, o);
    count += __shfl_down_sync(0xffffffffu, count, o);
  }
  if (lane == 0) {
    sp[warp] = p;
    sn[warp] = count;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kBinThreads / 32; ++w) {
      p += sp[w];
      count += sn[w];
    }
    part_p[(int64_t)blockIdx.y * nbins + b] = p;
    part_n[(int64_t)blockIdx.y * nbins + b] = (double)count;
  }
}

// All bins at once, where a warp's histogram fits the shared memory: warps take rows
// along x (read once, coalesced), along which the bin does not decrease, so a warp adds
// the modes of a bin by shuffles between neighbouring lanes and the first lane of each
// run adds the total to the warp's own histogram: nothing atomic, and a fixed order.
// 256^3 FP32: 137 us, 212 for the kernel above, which reads single modes out of 32-byte
// sectors; latency of the shuffles and of the histogram bounds it (HBM: 10 us), and
// eight blocks an SM in place of four are no faster.  A whole spectrum at 256^3 FP32:
// 761 -> 291 us, 64^3 173 -> 60, 4096^2 694 -> 317, 65536 161 -> 77.
template <typename T>
struct RowSum;
template <>
struct RowSum<float> {
  static constexpr int bytes = 12;   // a pair and a count per bin and warp
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void take(const PowerSum& p) {
    hi = p.hi;
    lo = p.lo;
  }
  __device__ __forceinline__ void add_lane(int o, bool same) {
    const float h = __shfl_down_sync(0xffffffffu, hi, o), l = __shfl_down_sync(0xffffffffu, lo, o);
    if (same) {
      lo += l;
      ce::add_to(hi, lo, h);
    }
  }
  __device__ __forceinline__ void add_to_bin(float2* bin) const {
    float2 x = *bin;
    x.y += lo;
    ce::add_to(x.x, x.y, hi);
    *bin = x;
  }
  static __device__ __forceinline__ double value(const float2& x) { return (double)x.x + (double)x.y; }
  using Bin = float2;
};
template <>
struct RowSum<double> {
  static constexpr int bytes = 12;
  double v = 0.0;
  __device__ __forceinline__ void take(const PowerSum& p) { v = p.wide; }
  __device__ __forceinline__ void add_lane(int o, bool same) {
    const double x = __shfl_down_sync(0xffffffffu, v, o);
    if (same) v += x;
  }
  __device__ __forceinline__ void add_to_bin(double* bin) const { *bin += v; }
  static __device__ __forceinline__ double value(double x) { return x; }
  using Bin = double;
};

constexpr int kBinWarps = kBinThreads / 32;
inline size_t rows_smem(int nbins) { return (size_t)nbins * (8 + kBinWarps * 12); }

template <typename C, typename T>
__global__ void __launch_bounds__(kBinThreads) k_bin_rows(const C* __restrict__ F, const T* __restrict__ f, int N,
                                                           int dims, int nbins, double* __restrict__ part_p,
                                                           double* __restrict__ part_n) {
  using Bin = typename RowSum<T>::Bin;
  extern __shared__ __align__(16) unsigned char hist[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double* wide = reinterpret_cast<double*>(hist);            // values outside the pairs' range, the whole block's
  Bin* bins = reinterpret_cast<Bin*>(wide + nbins);          // [warp][bin]
  unsigned* counts = reinterpret_cast<unsigned*>(bins + (size_t)kBinWarps * nbins);
  for (int b = threadIdx.x; b < nbins; b += kBinThreads) wide[b] = 0.0;
  for (int b = threadIdx.x; b < kBinWarps * nbins; b += kBinThreads) {
    bins[b] = Bin{};
    counts[b] = 0u;
  }
  __syncthreads();
  Bin* mine = bins + (size_t)warp * nbins;
  unsigned* mine_n = counts + (size_t)warp * nbins;
  const int half = N / 2, nx = half + 1, rows = dims == 3 ? N * N : N;
  const double sites = (double)N * (double)N * (dims == 3 ? (double)N : 1.0);
  for (int row = blockIdx.x * kBinWarps + warp; row < rows; row += gridDim.x * kBinWarps) {
    int ny = row % N, nz = row / N;
    ny = ny <= half ? ny : ny - N;
    nz = nz <= half ? nz : nz - N;
    const int r2 = ny * ny + nz * nz;
    const C* at = F + (int64_t)row * nx;
    for (int x0 = 0; x0 <= half; x0 += 32) {
      const int ix = x0 + lane, n2 = r2 + ix * ix, root = isqrt(n2);
      const int b = ix <= half ? root + (n2 > root * root + root) : 0x7fffffff;
      const bool in = b < nbins;
      const int w = ix == 0 || (N % 2 == 0 && ix == half) ? 1 : 2;
      PowerSum p;
      if (in) {
        const C v = at[ix];
        if (n2 == 0) p.add((double)v.x + (double)f[0] * sites, (double)v.y, 1.0);   // S f(site 0)
        else p.add(v.x, v.y, (decltype(v.x))w);
        if (sizeof(T) == 4 && p.wide != 0.0) atomicAdd(wide + b, p.wide);   // also NaN
      }
      RowSum<T> s;
      s.take(p);
      int n = in ? w : 0;
      for (int o = 1; o < 32; o *= 2) {
        const int other = __shfl_down_sync(0xffffffffu, b, o);
        const bool same = lane + o < 32 && other == b;
        if (!__any_sync(0xffffffffu, same)) break;
        s.add_lane(o, same);
        const int m = __shfl_down_sync(0xffffffffu, n, o);
        n += same ? m : 0;
      }
      const int before = __shfl_up_sync(0xffffffffu, b, 1);
      if (in && (lane == 0 || before != b)) {
        s.add_to_bin(mine + b);
        mine_n[b] += (unsigned)n;
      }
      __syncwarp();   // the next 32 modes may begin in this bin
      if (__shfl_sync(0xffffffffu, b, 31) >= nbins) break;   // no later mode of the row is in a bin
    }
  }
  __syncthreads();
  for (int b = threadIdx.x; b < nbins; b += kBinThreads) {
    double p = wide[b], n = 0.0;
    for (int w = 0; w < kBinWarps; ++w) {
      p += RowSum<T>::value(bins[(size_t)w * nbins + b]);
      n += (double)counts[(size_t)w * nbins + b];
    }
    part_p[(int64_t)blockIdx.x * nbins + b] = p;
    part_n[(int64_t)blockIdx.x * nbins + b] = n;
  }
}

// Bins the half spectrum F into `parts` partial histograms of nbins (at most kBinParts).
template <typename C, typename T>
cudaError_t bin_spectrum(cudaStream_t st, int sms, const void* F, const void* f, int64_t N, int dims, int nbins,
                         double* part_p, double* part_n, int* parts) {
  const C* Fc = static_cast<const C*>(F);
  const T* ft = static_cast<const T*>(f);
  // n^2 <= dims (N/2)^2, and b^2 + b a little above: exact in a float?
  const bool small = (double)dims * (double)(N / 2 + 2) * (double)(N / 2 + 2) < 16e6;
  const size_t shm = rows_smem(nbins);
  if (dims >= 2 && small && shm <= kRowsSmem) {
    const int rows = (int)(dims == 3 ? N * N : N);
    const int per_sm = (int)std::max<size_t>(1, std::min<size_t>(4, kRowsSmem / shm));
    *parts = std::min(std::min(kBinParts, per_sm * sms), (rows + kBinWarps - 1) / kBinWarps);
    const cudaError_t e = cudaFuncSetAttribute(k_bin_rows<C, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowsSmem);
    if (e != cudaSuccess) return e;
    k_bin_rows<C, T><<<*parts, kBinThreads, shm, st>>>(Fc, ft, (int)N, dims, nbins, part_p, part_n);
    return cudaGetLastError();
  }
  // rows of a bin per block: eight planes' worth of nz (3D), 1024 rows (2D)
  *parts = dims == 1 ? 1 : (int)std::min<int64_t>(kBinChunks, dims == 3 ? (N + 31) / 32 : (N + 1023) / 1024);
  const dim3 grid(nbins, *parts);
  if (small) k_bin_spectrum<C, T, int><<<grid, kBinThreads, 0, st>>>(Fc, ft, N, dims, nbins, part_p, part_n);
  else k_bin_spectrum<C, T, int64_t><<<grid, kBinThreads, 0, st>>>(Fc, ft, N, dims, nbins, part_p, part_n);
  return cudaGetLastError();
}

// One warp per bin: lanes take parts l, l + 32, ..., then a fixed shuffle tree.
__global__ void k_spectrum_finalize(const double* __restrict__ part_p, const double* __restrict__ part_n, int parts,
                                    int nbins, double* __restrict__ p_out, double* __restrict__ n_out) {
  const int lane = threadIdx.x & 31, b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (b >= nbins) return;
  double p = 0.0, n = 0.0;
  for (int k = lane; k < parts; k += 32) {
    p += part_p[(int64_t)k * nbins + b];
    n += part_n[(int64_t)k * nbins + b];
  }
  p = ce::warp_sum(p);
  n = ce::warp_sum(n);
  if (lane == 0) {
    p_out[b] = n > 0.0 ? p / n : 0.0;
    n_out[b] = n;
  }
}

struct SpectrumWork {
  cufftHandle plan = 0;
  bool have_plan = false;
  void* spec = nullptr;      // complex half spectrum
  void* real = nullptr;      // f - f(site 0), the transform's input
  double* part = nullptr;    // per-block histograms (2 x blocks x nbins_max)
  double* out = nullptr;     // 2 x nbins_max
  int nbins_max = 0;
};

std::vector<std::pair<const ce_sim*, SpectrumWork>>& work_table() {
  static std::vector<std::pair<const ce_sim*, SpectrumWork>> t;
  return t;
}

SpectrumWork* find_work(const ce_sim* s, bool create) {
  for (auto& e : work_table())
    if (e.first == s) return &e.second;
  if (!create) return nullptr;
  work_table().push_back({s, SpectrumWork{}});
  return &work_table().back().second;
}

// Partial histograms a handle's work buffers hold.
int spectrum_parts(const ce_sim* s) { return s->dims == 1 ? 1 : kBinParts; }

constexpr char kMagic[8] = {'C', 'E', 'G', 'R', 'I', 'D', '0', '1'};

struct FileHeader {
  char magic[8];
  int32_t dims, nfields, precision, expansion;
  int64_t N;
  double L, dt, q[3], kappa2;
  double a, ap_half, app, t;
  int64_t step;
};

}  // namespace

// Release the spectrum work buffers of a handle (called from ce_free).
void ce::outputs_release(const ce_sim* s) {
  auto& t = work_table();
  for (size_t i = 0; i < t.size(); ++i) {
    if (t[i].first != s) continue;
    SpectrumWork& w = t[i].second;
    if (w.have_plan) cufftDestroy(w.plan);
    if (w.spec) cudaFree(w.spec);
    if (w.real) cudaFree(w.real);
    if (w.part) cudaFree(w.part);
    if (w.out) cudaFree(w.out);
    t.erase(t.begin() + (long)i);
    return;
  }
}

extern "C" {

int ce_spectrum(ce_sim* s, int field, int nbins, double* k, double* power, double* count) {
  ce::set_last_error("");
  if (!s) return ofail(CE_EINVAL, "ce_spectrum: sim is NULL");
  if (!k || !power || !count) return ofail(CE_EINVAL, "ce_spectrum: NULL output");
  if (field < 0 || field >= s->nf) return ofail(CE_EINVAL, "ce_spectrum: field out of range");
  if (!s->have_state) return ofail(CE_ESTATE, "ce_spectrum: no fields set");
  const int max_bins = (int)std::ceil(std::sqrt((double)s->dims) * (double)(s->N / 2)) + 2;
  if (nbins < 1 || nbins > max_bins)
    return ofail(CE_EINVAL, "ce_spectrum: nbins must be 1..ceil(sqrt(dims) N/2) + 2");
  cudaError_t e = cudaSetDevice(s->device);
  if (e == cudaSuccess && s->batch) e = ce::batch_wait(s->batch);
  if (e != cudaSuccess) return ocuda(e, "ce_spectrum");
  SpectrumWork* w = find_work(s, true);
  const bool f32 = s->prec == CE_F32;
  int64_t half = s->N / 2 + 1;
  for (int d = 1; d < s->dims; ++d) half *= s->N;
  if (!w->have_plan) {
    int n[3] = {(int)s->N, (int)s->N, (int)s->N};
    cufftResult r = cufftPlanMany(&w->plan, s->dims, n, nullptr, 1, 0, nullptr, 1, 0, f32 ? CUFFT_R2C : CUFFT_D2Z, 1);
    if (r != CUFFT_SUCCESS) return ofail(CE_ECUDA, "ce_spectrum: cufft plan failed");
    w->have_plan = true;
    e = cudaMalloc(&w->spec, (size_t)half * (f32 ? sizeof(cufftComplex) : sizeof(cufftDoubleComplex)));
    if (e == cudaSuccess) e = cudaMalloc(&w->real, (size_t)s->S * s->esize);
    if (e == cudaSuccess) e = cudaMalloc(&w->part, sizeof(double) * 2 * spectrum_parts(s) * max_bins);
    if (e == cudaSuccess) e = cudaMalloc(&w->out, sizeof(double) * 2 * max_bins);
    if (e != cudaSuccess) {
      ce::outputs_release(s);
      return ofail(CE_ENOMEM, "ce_spectrum: work buffers");
    }
    w->nbins_max = max_bins;
  }
  cufftSetStream(w->plan, s->stream);
  const int cblocks = (int)std::min<int64_t>((s->S + 255) / 256, (int64_t)s->sms * 8);
  if (f32)
    k_shifted_copy<float><<<cblocks, 256, 0, s->stream>>>(static_cast<const float*>(s->f[s->cur][field]),
                                                           static_cast<float*>(w->real), s->S);
  else
    k_shifted_copy<double><<<cblocks, 256, 0, s->stream>>>(static_cast<const double*>(s->f[s->cur][field]),
                                                            static_cast<double*>(w->real), s->S);
  e = cudaGetLastError();
  if (e != cudaSuccess) return ocuda(e, "ce_spectrum: shift");
  cufftResult r;
  if (f32)
    r = cufftExecR2C(w->plan, static_cast<cufftReal*>(w->real), static_cast<cufftComplex*>(w->spec));
  else
    r = cufftExecD2Z(w->plan, static_cast<cufftDoubleReal*>(w->real), static_cast<cufftDoubleComplex*>(w->spec));
  if (r != CUFFT_SUCCESS) return ofail(CE_ECUDA, "ce_spectrum: cufft exec failed");
  double* part_p = w->part;
  double* part_n = w->part + (int64_t)spectrum_parts(s) * nbins;
  int parts = 1;
  const void* field_data = s->f[s->cur][field];
  e = f32 ? bin_spectrum<cufftComplex, float>(s->stream, s->sms, w->spec, field_data, s->N, s->dims, nbins, part_p,
                                              part_n, &parts)
          : bin_spectrum<cufftDoubleComplex, double>(s->stream, s->sms, w->spec, field_data, s->N, s->dims, nbins,
                                                     part_p, part_n, &parts);
  if (e != cudaSuccess) return ocuda(e, "ce_spectrum: binning");
  k_spectrum_finalize<<<(nbins + 7) / 8, 256, 0, s->stream>>>(part_p, part_n, parts, nbins, w->out, w->out + nbins);
  std::vector<double> host(2 * (size_t)nbins);
  e = cudaMemcpyAsync(host.data(), w->out, sizeof(double) * 2 * nbins, cudaMemcpyDeviceToHost, s->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  if (e != cudaSuccess) return ocuda(e, "ce_spectrum: read-back");
  const double two_pi_over_L = 2.0 * M_PI / s->cfg.L;
  for (int b = 0; b < nbins; ++b) {
    k[b] = two_pi_over_L * b;
    power[b] = host[b];
    count[b] = host[nbins + b];
  }
  return CE_OK;
}

int ce_sample_fields(ce_sim* s, const int64_t* sites, int64_t n, double* f, double* v, ce_scalars_t* sc) {
  ce::set_last_error("");
  if (!s) return ofail(CE_EINVAL, "ce_sample_fields: sim is NULL");
  if (n < 0 || (n > 0 && (!sites || !f || !v)) || !sc) return ofail(CE_EINVAL, "ce_sample_fields: bad arguments");
  if (!s->have_state) return ofail(CE_ESTATE, "ce_sample_fields: no fields set");
  for (int64_t k = 0; k < n; ++k)
    if (sites[k] < 0 || sites[k] >= s->S) return ofail(CE_EINVAL, "ce_sample_fields: site index out of range");
  cudaError_t e = cudaSetDevice(s->device);
  if (e == cudaSuccess && s->batch) e = ce::batch_wait(s->batch);
  if (e != cudaSuccess) return ocuda(e, "ce_sample_fields");
  // the staging buffer (chunk x nf doubles) holds, per pass, m site indices and
  // the m x nf values of f and of v
  const int64_t cap = s->chunk * s->nf * 8;
  const int64_t mmax = std::max<int64_t>(1, cap / (8 + 16 * (int64_t)s->nf));
  unsigned char* stage = reinterpret_cast<unsigned char*>(s->staging);
  const void* slot = &s->aux->slot[s->cur];
  for (int64_t k0 = 0; k0 < n; k0 += mmax) {
    const int64_t m = std::min<int64_t>(mmax, n - k0);
    int64_t* d_sites = reinterpret_cast<int64_t*>(stage);
    double* d_f = reinterpret_cast<double*>(stage + m * 8);
    double* d_v = d_f + m * s->nf;
    e = cudaMemcpyAsync(d_sites, sites + k0, (size_t)m * 8, cudaMemcpyHostToDevice, s->stream);
    if (e != cudaSuccess) return ocuda(e, "ce_sample_fields: site upload");
    const int blocks = (int)std::min<int64_t>((m + 255) / 256, (int64_t)s->sms * 4);
    if (s->prec == CE_F32) {
      SamplePtrs<float> p{};
      for (int i = 0; i < s->nf; ++i) {
        p.f[i] = static_cast<const float*>(s->f[s->cur][i]);
        p.w[i] = static_cast<const float*>(s->w[s->cur][i]);
      }
      k_sample<float><<<blocks, 256, 0, s->stream>>>(p, s->nf, static_cast<const ce::DevScalars*>(slot), d_sites, m,
                                                     d_f, d_v);
    } else {
      SamplePtrs<double> p{};
      for (int i = 0; i < s->nf; ++i) {
        p.f[i] = static_cast<const double*>(s->f[s->cur][i]);
        p.w[i] = static_cast<const double*>(s->w[s->cur][i]);
      }
      k_sample<double><<<blocks, 256, 0, s->stream>>>(p, s->nf, static_cast<const ce::DevScalars*>(slot), d_sites, m,
                                                      d_f, d_v);
    }
    e = cudaGetLastError();
    for (int i = 0; i < s->nf && e == cudaSuccess; ++i) {
      e = cudaMemcpyAsync(f + (int64_t)i * n + k0, d_f + (int64_t)i * m, (size_t)m * 8, cudaMemcpyDeviceToHost,
                          s->stream);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(v + (int64_t)i * n + k0, d_v + (int64_t)i * m, (size_t)m * 8, cudaMemcpyDeviceToHost,
                            s->stream);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    if (e != cudaSuccess) return ocuda(e, "ce_sample_fields: gather");
  }
  ce::DevAux host{};
  e = cudaMemcpyAsync(&host, s->aux, sizeof(host), cudaMemcpyDeviceToHost, s->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  if (e != cudaSuccess) return ocuda(e, "ce_sample_fields: scalars");
  if (host.status != CE_OK) return ofail(host.status, "ce_sample_fields: the device reported an error");
  const ce::DevScalars& d = host.slot[s->cur];
  sc->a = s->cfg.expansion ? d.a : 1.0;
  sc->ap_half = s->cfg.expansion ? d.ap : 0.0;
  sc->app = s->cfg.expansion ? d.app : 0.0;
  sc->t = s->t;
  sc->step = s->step;
  return CE_OK;
}

int ce_save(ce_sim* s, const char* path) {
  ce::set_last_error("");
  if (!s || !path) return ofail(CE_EINVAL, "ce_save: NULL argument");
  if (!s->have_state) return ofail(CE_ESTATE, "ce_save: no fields set");
  const size_t n = (size_t)s->nf * (size_t)s->S;
  std::vector<double> f(n), v(n);
  ce_scalars_t sc;
  int rc = ce_get_fields(s, f.data(), v.data(), CE_VEL_STAGGERED, &sc);
  if (rc != CE_OK) return rc;
  FileHeader h;
  std::memset(&h, 0, sizeof(h));
  std::memcpy(h.magic, kMagic, 8);
  h.dims = s->dims;
  h.nfields = s->nf;
  h.precision = s->prec;
  h.expansion = s->cfg.expansion;
  h.N = s->N;
  h.L = s->cfg.L;
  h.dt = s->cfg.dt;
  for (int i = 0; i < 3; ++i) h.q[i] = s->cfg.q[i];
  h.kappa2 = s->kappa2;
  h.a = sc.a;
  h.ap_half = sc.ap_half;
  h.app = sc.app;
  h.t = sc.t;
  h.step = sc.step;
  FILE* fp = std::fopen(path, "wb");
  if (!fp) return ofail(CE_EINVAL, std::string("ce_save: cannot open ") + path);
  bool ok = std::fwrite(&h, sizeof(h), 1, fp) == 1 && std::fwrite(f.data(), sizeof(double), n, fp) == n &&
            std::fwrite(v.data(), sizeof(double), n, fp) == n;
  ok = (std::fclose(fp) == 0) && ok;
  return ok ? CE_OK : ofail(CE_EINVAL, std::string("ce_save: write failed for ") + path);
}

int ce_load(ce_sim* s, const char* path) {
  ce::set_last_error("");
  if (!s || !path) return ofail(CE_EINVAL, "ce_load: NULL argument");
  FILE* fp = std::fopen(path, "rb");
  if (!fp) return ofail(CE_EINVAL, std::string("ce_load: cannot open ") + path);
  FileHeader h;
  if (std::fread(&h, sizeof(h), 1, fp) != 1 || std::memcmp(h.magic, kMagic, 8) != 0) {
    std::fclose(fp);
    return ofail(CE_EINVAL, "ce_load: not a grid image");
  }
  if (h.dims != s->dims || h.N != s->N || h.nfields != s->nf || h.expansion != s->cfg.expansion ||
      h.L != s->cfg.L || h.dt != s->cfg.dt || h.q[0] != s->cfg.q[0] || h.q[1] != s->cfg.q[1] ||
      h.q[2] != s->cfg.q[2] || h.kappa2 != s->kappa2) {
    std::fclose(fp);
    return ofail(CE_EINVAL, "ce_load: the image was written for another lattice or model");
  }
  const size_t n = (size_t)s->nf * (size_t)s->S;
  std::vector<double> f(n), v(n);
  const bool ok = std::fread(f.data(), sizeof(double), n, fp) == n && std::fread(v.data(), sizeof(double), n, fp) == n;
  std::fclose(fp);
  if (!ok) return ofail(CE_EINVAL, "ce_load: truncated image");
  ce_scalars_t sc{h.a, h.ap_half, h.app, h.t, h.step};
  return ce_set_fields(s, f.data(), v.data(), CE_VEL_STAGGERED, &sc);
}

}  // extern "C"
