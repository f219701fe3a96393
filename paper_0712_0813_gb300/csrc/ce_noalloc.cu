// ce_noalloc.cu -- ce_moments_noalloc: per-field mean and variance of field
// arrays the caller already holds in device memory, computed without any
// device allocation by the library.
//
// Scratch lives in one file-scope __device__ array (g_moments_scratch, 64 KiB)
// that every GPU loading the library keeps until the process exits.  Host code
// must not hand the array's name to a kernel (on the host it is only a
// stand-in for the symbol), so the device address is fetched once per device
// with cudaGetSymbolAddress and passed to the kernels explicitly.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <mutex>
#include <string>

#include "ce_internal.h"
#include "clusterlat.h"

namespace {

constexpr int kBlocks = 1024;          // most blocks per field of the partial-sum pass (size of the scratch)
constexpr int kBatch = 8;              // loads a thread has in flight
constexpr int64_t kPairsMin = int64_t(1) << 17;   // FP32 arrays from this size take k_moments_partial_pairs
constexpr int kThreads = 256;
constexpr int kMaxFields = 4;
constexpr int kMaxDevices = 64;
constexpr int64_t kMaxSites = int64_t(1) << 34;

// Partial sums, [block][field][2]: sum (f - f0) and sum (f - f0)^2 with
// f0 = the field's first value.  Every call overwrites the slots it reads, so
// nothing here has to start at zero.
static __device__ __align__(256) double g_moments_scratch[kBlocks * kMaxFields * 2];

std::mutex g_setup_mutex;
double* g_scratch_ptr[kMaxDevices] = {};

int noalloc_fail(int code, const std::string& msg) {
  ce::set_last_error(msg);
  return code;
}

// Device address of the scratch array for the current device (set-up once per device).
int scratch_for_device(int dev, double** out) {
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_moments_scratch);
    if (e != cudaSuccess || !p)
      return noalloc_fail(CE_ECUDA, std::string("ce_moments_noalloc: cudaGetSymbolAddress failed: ") +
                                        cudaGetErrorString(e));
    g_scratch_ptr[dev] = static_cast<double*>(p);
  }
  *out = g_scratch_ptr[dev];
  return CE_OK;
}

// hi + lo += x: the addition's rounding error (Knuth's TwoSum, exact) joins lo.  Intrinsics,
// which the compiler does not contract with a product that x may be: else what is added
// would depend on the code around.
__device__ __forceinline__ void add_to(float& hi, float& lo, float x) {
  const float s = __fadd_rn(hi, x);
  const float b = __fsub_rn(s, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(x, b)));
  hi = s;
}

// Block sums of (f - f0) and (f - f0)^2, FP32 arrays; blockIdx.y is the field.
//
// The sums carry FP64 accuracy without the FP64 pipe (two lanes per clock and
// SM against 128 FP32 lanes): f - f0 is split exactly into dh + dl and its square
// into p + pe + dl^2 (pe = the FMA residual of dh^2, plus 2 dh dl), and dh, p and
// pe are each summed as an unevaluated pair of floats (add_to).  A single pair for
// p and pe was not enough: rounding pe into the low word left a bias of 1e-15 of
// the sum.  Now a sum is within ~1e-17 of the exact one for 2^17 sites and more;
// smaller arrays take the FP64 form below, latency is all they pay for.  The
// lanes' pairs are added the same way and only the warps' are converted.  Elements
// whose square or its residual would leave FP32's range (|dh| below 2^-40, or 2^50
// and above, infinities and NaN) go to FP64 sums in a branch of its own: if-converted
// into the loop, its FP64 operations cost as much as the FP64 form.
// Four 128^3 fields took 198 us with FP64 per element (conversion, subtraction,
// addition and FMA: 4 x 64 cycles a warp and scheduler), the fields one after
// another and a last pass of one thread per field.
__global__ void __launch_bounds__(kThreads) k_moments_partial_pairs(const float* __restrict__ f, int64_t n,
                                                                    double* __restrict__ scratch) {
  constexpr int kWords = 4;
  __shared__ float red[2][kThreads / 32][kWords + 1];
  __shared__ double redd[2][kThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  const float* fi = f + (int64_t)blockIdx.y * n;
  const float f0 = fi[0];
  float a = 0.f, al = 0.f, ad = 0.f;                       // sum of dh (pair), of dl
  float b = 0.f, bl = 0.f, c = 0.f, cl = 0.f, bt = 0.f;    // of p (pair), pe (pair), dl^2
  double wa = 0.0, wb = 0.0;                               // elements outside the pairs' range
  bool wide = false;
  for (int64_t base = (int64_t)blockIdx.x * kThreads; base < n; base += kBatch * stride) {
    const int64_t k0 = base + threadIdx.x;
    float xs[kBatch];   // positions past the end repeat f0, which adds nothing
    bool odd = false;
#pragma unroll
    for (int r = 0; r < kBatch; ++r) xs[r] = k0 + r * stride < n ? __ldg(fi + k0 + r * stride) : f0;
#pragma unroll
    for (int r = 0; r < kBatch; ++r) {
      const float x = xs[r];
      float dh = x - f0;
      const float t = dh - x;
      float dl = (x - (dh - t)) + (-f0 - t);
      const float mag = fabsf(dh);
      if (!((mag >= 0x1p-40f && mag < 0x1p50f) || x == f0)) {
        odd = true;
        dh = dl = 0.f;
      }
      const float p = __fmul_rn(dh, dh);
      const float pe = fmaf(2.f * dh, dl, fmaf(dh, dh, -p));
      add_to(a, al, dh);
      ad += dl;
      add_to(b, bl, p);
      add_to(c, cl, pe);
      bt = fmaf(dl, dl, bt);
    }
    if (__any_sync(0xffffffffu, odd)) {
      wide = true;
#pragma unroll 1
      for (int r = 0; r < kBatch; ++r) {
        const int64_t k = k0 + r * stride;
        const float x = k < n ? __ldg(fi + k) : f0;
        const float mag = fabsf(x - f0);
        if (!((mag >= 0x1p-40f && mag < 0x1p50f) || x == f0)) {
          const double d = (double)x - (double)f0;
          wa += d;
          wb += d * d;
        }
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    al += __shfl_down_sync(0xffffffffu, al, o);
    ad += __shfl_down_sync(0xffffffffu, ad, o);
    bl += __shfl_down_sync(0xffffffffu, bl, o);
    cl += __shfl_down_sync(0xffffffffu, cl, o);
    bt += __shfl_down_sync(0xffffffffu, bt, o);
    add_to(a, al, __shfl_down_sync(0xffffffffu, a, o));
    add_to(b, bl, __shfl_down_sync(0xffffffffu, b, o));
    add_to(c, cl, __shfl_down_sync(0xffffffffu, c, o));
  }
  if (wide) {   // the same for the whole warp
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      wa += __shfl_down_sync(0xffffffffu, wa, o);
      wb += __shfl_down_sync(0xffffffffu, wb, o);
    }
  }
  if (lane == 0) {
    const float qa[kWords] = {a, al, ad, 0.f}, qb[kWords] = {b, c, bl, cl + bt};
#pragma unroll
    for (int j = 0; j < kWords; ++j) {
      red[0][warp][j] = qa[j];
      red[1][warp][j] = qb[j];
    }
    redd[0][warp] = wa;
    redd[1][warp] = wb;
  }
  __syncthreads();
  // thread (q, w) = (t / 8, t % 8): warp w's sum of quantity q, then a tree over the 8 warps
  static_assert(kThreads == 256, "the sum over the warps below is written for 8 of them");
  if (threadIdx.x < 16) {
    const int q = threadIdx.x >> 3, w = threadIdx.x & 7;
    double v = redd[q][w];
#pragma unroll
    for (int j = kWords - 1; j >= 0; --j) v += (double)red[q][w][j];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_down_sync(0xffffu, v, o, 8);
    if (w == 0) scratch[((int64_t)blockIdx.x * kMaxFields + blockIdx.y) * 2 + q] = v;
  }
}

// The same with FP64 sums: FP64 arrays, and FP32 arrays too small for the pairs'
// errors to average out.
template <typename T>
__global__ void __launch_bounds__(kThreads) k_moments_partial(const T* __restrict__ f, int64_t n,
                                                              double* __restrict__ scratch) {
  __shared__ double red[kThreads / 32][2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  const T* fi = f + (int64_t)blockIdx.y * n;
  const T f0 = fi[0];
  const double shift = (double)f0;
  double s1 = 0.0, s2 = 0.0;
  for (int64_t k0 = (int64_t)blockIdx.x * kThreads + threadIdx.x; k0 < n; k0 += kBatch * stride) {
    T xs[kBatch];
#pragma unroll
    for (int r = 0; r < kBatch; ++r) xs[r] = k0 + r * stride < n ? __ldg(fi + k0 + r * stride) : f0;
#pragma unroll
    for (int r = 0; r < kBatch; ++r) {
      const double d = (double)xs[r] - shift;
      s1 += d;
      s2 += d * d;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s1 += __shfl_down_sync(0xffffffffu, s1, o);
    s2 += __shfl_down_sync(0xffffffffu, s2, o);
  }
  if (lane == 0) {
    red[warp][0] = s1;
    red[warp][1] = s2;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double t = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) t += red[w][threadIdx.x];
    scratch[((int64_t)blockIdx.x * kMaxFields + blockIdx.y) * 2 + threadIdx.x] = t;
  }
}

// One block per field adds the `blocks` partial sums in a fixed order (thread t
// takes blocks t, t + 256, ..., then a fixed tree).
template <typename T>
__global__ void __launch_bounds__(kThreads) k_moments_final(const T* __restrict__ f, int64_t n, int blocks,
                                                            const double* __restrict__ scratch,
                                                            double* __restrict__ mean, double* __restrict__ var) {
  __shared__ double red[kThreads / 32][2];
  const int i = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double a = 0.0, b = 0.0;
  for (int blk = threadIdx.x; blk < blocks; blk += kThreads) {
    a += scratch[((int64_t)blk * kMaxFields + i) * 2];
    b += scratch[((int64_t)blk * kMaxFields + i) * 2 + 1];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
  }
  if (lane == 0) {
    red[warp][0] = a;
    red[warp][1] = b;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  a = b = 0.0;
  for (int w = 0; w < kThreads / 32; ++w) {
    a += red[w][0];
    b += red[w][1];
  }
  const double m1 = a / (double)n, m2 = b / (double)n;
  mean[i] = (double)f[(int64_t)i * n] + m1;
  var[i] = m2 - m1 * m1;
}

}  // namespace

extern "C" int ce_moments_noalloc(const void* f, int precision, int64_t n, int nfields, void* stream,
                                  double* mean, double* var) {
  ce::set_last_error("");
  if (!f || !mean || !var) return noalloc_fail(CE_EINVAL, "ce_moments_noalloc: NULL pointer");
  if (precision != CE_F32 && precision != CE_F64)
    return noalloc_fail(CE_EINVAL, "ce_moments_noalloc: precision must be CE_F32 or CE_F64");
  if (nfields < 1 || nfields > kMaxFields)
    return noalloc_fail(CE_EINVAL, "ce_moments_noalloc: nfields must be 1..4 (the static scratch holds 4 fields)");
  if (n < 1 || n > kMaxSites)
    return noalloc_fail(CE_EINVAL, "ce_moments_noalloc: n must be 1..2^34 sites per field");
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return noalloc_fail(CE_ECUDA, std::string("ce_moments_noalloc: ") + cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return noalloc_fail(CE_EINVAL, "ce_moments_noalloc: device index out of range");
  double* scratch = nullptr;
  int rc = scratch_for_device(dev, &scratch);
  if (rc != CE_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int64_t want = (n + (int64_t)kThreads * kBatch - 1) / ((int64_t)kThreads * kBatch);
  // about two waves of 8 resident blocks an SM over all fields
  const int cap = std::min(kBlocks, std::max(1, 16 * ce::sm_count(dev) / nfields));
  const int blocks = (int)std::min<int64_t>(want, cap);
  const dim3 grid(blocks, nfields);
  if (precision == CE_F32) {
    const float* ff = static_cast<const float*>(f);
    if (n >= kPairsMin) k_moments_partial_pairs<<<grid, kThreads, 0, st>>>(ff, n, scratch);
    else k_moments_partial<float><<<grid, kThreads, 0, st>>>(ff, n, scratch);
    k_moments_final<float><<<nfields, kThreads, 0, st>>>(ff, n, blocks, scratch, mean, var);
  } else {
    const double* fd = static_cast<const double*>(f);
    k_moments_partial<double><<<grid, kThreads, 0, st>>>(fd, n, scratch);
    k_moments_final<double><<<nfields, kThreads, 0, st>>>(fd, n, blocks, scratch, mean, var);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return noalloc_fail(CE_ECUDA, std::string("ce_moments_noalloc: launch: ") + cudaGetErrorString(e));
  return CE_OK;
}
