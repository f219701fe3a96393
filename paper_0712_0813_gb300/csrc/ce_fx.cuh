// ce_fx.cuh -- the FP64 step's force in integer arithmetic.
//
// GB300 issues one FP64 warp instruction per 64 cycles and scheduler (two lanes
// per clock and SM), an integer one every cycle or two.  The Laplacian and the
// model force of a site, 29 of the FP64 step's ~32 operations a site with two
// fields, are therefore formed on 64-bit integers; FP64 keeps the drift, the kick
// and one addition to the energy sums.
//
// An Fx is a double's 53-bit significand left-justified in 58 bits of a signed
// integer with the double's own exponent (exact for every finite double).  A
// site's neighbours are aligned to the largest exponent among them, so what
// alignment drops of each is below 2^-57 of the largest value of the stencil, where
// FP64 rounds every partial sum to 2^-53 of it; products are the upper 64 bits of
// unsigned 64-bit fractions (7 instructions; a signed one takes 17), and the two meet
// in a unit 2^-54 of the model force or 2^-61 of the Laplacian.  The force is thus at
// least as accurate as FP64's, site by site, whatever the field's range.  Non-finite values are left to the caller (fx_finite).
//
// Plain C++ apart from the shift and the bit casts, so the CPU tests compile it.
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define CE_FX_HD __host__ __device__ __forceinline__
#else
#define CE_FX_HD inline
#endif

namespace ce {
namespace fx {

constexpr int kOne = 1080;      // Fx value = m 2^(e - 1080)
constexpr int kNonFinite = 2047;

struct Fx {
  int64_t m;   // |m| < 2^58
  int e;       // biased exponent of the double (1 for zero and subnormals)
};

// A positive constant (or zero) as a 64-bit fraction: value = m 2^(e - 64).
struct FxConst {
  uint64_t m;
  int e;
};

// Constants of one lattice: dx^2, q_i and q_i dx^2.
struct FxModel {
  FxConst dx2, q[3], qdx2[3];
};

CE_FX_HD int64_t bits_of(double x) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(x);
#else
  int64_t b;
  std::memcpy(&b, &x, 8);
  return b;
#endif
}

CE_FX_HD double from_bits(int64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double x;
  std::memcpy(&x, &b, 8);
  return x;
#endif
}

// x >> s, s >= 0 of any size (PTX clamps the shift to 63).
CE_FX_HD int64_t asr(int64_t x, int s) {
#ifdef __CUDA_ARCH__
  int64_t r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
  return r;
#else
  return x >> (s > 63 ? 63 : s);
#endif
}

// x << s, s >= 0 of any size.
CE_FX_HD int64_t shl(int64_t x, int s) {
#ifdef __CUDA_ARCH__
  int64_t r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
  return r;
#else
  return s > 63 ? 0 : (int64_t)((uint64_t)x << s);
#endif
}

// x >> s, to nearest.
CE_FX_HD int64_t asr_round(int64_t x, int s) {
  const int64_t r = asr(x, s - 1 < 0 ? 0 : s - 1);
  return s > 0 ? (r + 1) >> 1 : r;
}

CE_FX_HD int clz64(uint64_t x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}

CE_FX_HD int clz32(int x) {
#ifdef __CUDA_ARCH__
  return __clz(x);
#else
  return x ? __builtin_clz((unsigned)x) : 32;
#endif
}

CE_FX_HD int imax(int a, int b) { return a > b ? a : b; }
CE_FX_HD int imin(int a, int b) { return a < b ? a : b; }

CE_FX_HD Fx from_double(double x) {
  const int64_t b = bits_of(x);
  const int hi = (int)(b >> 32);
  const int e = (hi >> 20) & 0x7ff;
  const int64_t frac = (b & 0xfffffffffffffLL) | (e != 0 ? 0x10000000000000LL : 0);
  const int64_t s = b >> 63;
  Fx r;
  r.m = ((frac << 5) ^ s) - s;
  r.e = e != 0 ? e : 1;
  return r;
}

// The double an Fx came from (0.0 for -0.0, else bit for bit).
CE_FX_HD double to_double(const Fx& x) {
  const int64_t s = x.m >> 63;
  const int64_t frac = ((x.m ^ s) - s) >> 5;
  const int64_t e = (frac & 0x10000000000000LL) ? x.e : 0;
  return from_bits((s & INT64_MIN) | (e << 52) | (frac & 0xfffffffffffffLL));
}

// x >> s of an unsigned value, s >= 0 of any size.
CE_FX_HD uint64_t lsr(uint64_t x, int s) {
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
  return r;
#else
  return s > 63 ? 0 : x >> s;
#endif
}

// (x >> s) of an unsigned value, to nearest, for s >= 1.
CE_FX_HD int64_t lsr_round(uint64_t x, int s) { return (int64_t)((lsr(x, s - 1) + 1) >> 1); }

// r 2^u as a double, to nearest, subnormal below the normal range.  RANGE: infinite
// above it (else the caller knows that r 2^u stays clear of that).
template <bool RANGE>
CE_FX_HD double scaled(int64_t r, int u) {
  const int64_t s = r >> 63;
  uint64_t a = (uint64_t)((r ^ s) - s);
  const int z = clz64(a);
  a <<= z & 63;
  const int eb = u - z + 63 + 1023;
  int64_t b = (int64_t)((a >> 11) + ((a >> 10) & 1)) + ((int64_t)(eb - 1) << 52);
  if (RANGE) b = eb >= kNonFinite ? 0x7ff0000000000000LL : b;
  b = z == 64 ? 0 : b;
  if (eb < 1) b = lsr_round(a, 12 - eb);   // in units of 2^-1074
  return from_bits(b | (s & INT64_MIN));
}

// The upper 64 bits of a product: the product of two 64-bit fractions.
CE_FX_HD uint64_t mul(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

// x of either sign times a fraction, rounded down.
CE_FX_HD int64_t mul_signed(uint64_t a, int64_t x) {
  return (int64_t)(mul(a, (uint64_t)x) - (a & (uint64_t)(x >> 63)));
}

// x or -x for mask 0 or -1.
CE_FX_HD int64_t negate_if(int64_t x, int64_t mask) { return (x ^ mask) - mask; }

// The largest exponent of each field's stencil.
template <int NF, int DIMS>
CE_FX_HD void stencil_exponents(const Fx (&g)[NF], const Fx (&nb)[NF][2 * DIMS], int (&em)[NF]) {
#pragma unroll
  for (int i = 0; i < NF; ++i) {
    em[i] = g[i].e;
#pragma unroll
    for (int j = 0; j < 2 * DIMS; ++j) em[i] = imax(em[i], nb[i][j].e);
  }
}

// The products of a site, as 64-bit fractions with binary exponents: |g_i| (x, ex),
// phi^2 (p2, ep), dx^2 |dV/df_i| (d, in units of 2^ud) and dx^2 sum_i g_i dV/df_i
// = 4 dx^2 V (w, ew).
template <int NF>
struct SiteModel {
  uint64_t x[NF], d[NF], w;
  int ex[NF], ud[NF], ew;
};

template <int NF, bool SUMS>
CE_FX_HD void site_model(const Fx (&g)[NF], const FxModel& k, SiteModel<NF>& s) {
  constexpr int kRoom = NF == 1 ? 0 : (NF == 2 ? 1 : 2);   // bits a sum of NF fractions may gain
#pragma unroll
  for (int i = 0; i < NF; ++i) {
    s.x[i] = (uint64_t)negate_if(g[i].m, g[i].m >> 63) << 6;
    s.ex[i] = g[i].e - 1022;
  }
  const uint64_t p2 = mul(s.x[0], s.x[0]);
  const int ep = 2 * s.ex[0];
  // t = phi^2 + sum_i q_i chi_i^2
  uint64_t pt = p2, t = p2;
  int et = ep;
  if constexpr (NF > 1) {
    uint64_t c[NF];
    int ec[NF];
#pragma unroll
    for (int i = 1; i < NF; ++i) {
      c[i] = mul(mul(s.x[i], s.x[i]), k.q[i - 1].m);
      ec[i] = 2 * s.ex[i] + k.q[i - 1].e;
      et = imax(et, ec[i]);
    }
    et += kRoom;
    pt = lsr(p2, et - ep);
    t = pt;
#pragma unroll
    for (int i = 1; i < NF; ++i) t += lsr(c[i], et - ec[i]);
  }
  // g_i (dx^2 t) for phi, g_i (q_i dx^2 phi^2) for the others
  s.d[0] = mul(s.x[0], mul(t, k.dx2.m));
  s.ud[0] = s.ex[0] + et + k.dx2.e - 64;
#pragma unroll
  for (int i = 1; i < NF; ++i) {
    s.d[i] = mul(s.x[i], mul(p2, k.qdx2[i - 1].m));
    s.ud[i] = s.ex[i] + ep + k.qdx2[i - 1].e - 64;
  }
  if constexpr (SUMS) {   // phi^2 (2 t - phi^2)
    s.w = mul(mul(p2, t - (pt >> 1)), k.dx2.m);
    s.ew = ep + et + 1 + k.dx2.e;
  }
}

// Whether the site may take site_force's fast form: finite values far from FP64's
// largest, and every dx^2 dV/df_i, and their sum with g_i, finer than raw_i by two
// bits and more (dx^2 V'' below about 4).
template <int NF>
CE_FX_HD bool fast_site(const int (&em)[NF], const SiteModel<NF>& s) {
  bool ok = true;
#pragma unroll
  for (int i = 0; i < NF; ++i) ok = ok && em[i] < 1023 + 200 && s.ud[i] + 2 < em[i] - kOne;
  return ok;
}

// A site's force over 1/dx^2 and its term of the energy sum that drives a(t).
//   force[i] = raw_i - dx^2 dV/df_i, raw_i = sum of the 2d neighbours - 2d g_i
//   energy   = sum_i g_i (raw_i - 3/4 dx^2 dV/df_i)
// With V = 1/4 sum_i f_i dV/df_i and, on a periodic lattice, sum_x |grad g|^2 =
// -dx^-2 sum_x g raw, the lattice sum of energy is -dx^2 S (2 G + 3 V): the one
// combination of the mean gradient and potential energies that a'' needs.
// g[i]: the site; nb[i][0 .. 2d - 1]: its neighbours.  flip: 0 or -1, rounds the
// energy terms with their signs turned: callers alternate it from lane to lane,
// so that what rounding downwards adds to the terms (1e-15 of the sum, as a bias)
// cancels over the lattice.
// raw is moved up to the 62 bits it may fill, as far as the model force's own unit
// allows, before the two meet: on a fine or smooth lattice raw is far below its
// operands, and in their unit (2^-57 of g) the model force of a homogeneous field was
// off by 2^-58 / dx^2, the same way at every site (1e-10 of it at dx^2 = 1e-7).
template <int NF, int DIMS, bool SUMS, bool FAST>
CE_FX_HD void site_force(const Fx (&g)[NF], const Fx (&nb)[NF][2 * DIMS], const int (&em)[NF],
                         const SiteModel<NF>& s, int flip, double (&force)[NF], double& energy) {
  constexpr int kRoom = NF <= 2 ? 1 : 2;
  int64_t z[NF];
  int uz[NF];
#pragma unroll
  for (int i = 0; i < NF; ++i) {
    const int64_t sign = g[i].m >> 63;
    // raw, aligned to the stencil's largest exponent
    int64_t raw = asr(g[i].m * (-2 * DIMS), em[i] - g[i].e);
#pragma unroll
    for (int j = 0; j < 2 * DIMS; ++j) raw += asr(nb[i][j].m, em[i] - nb[i][j].e);
    const int ur = em[i] - kOne;
    // |raw| <= 3 2^60: at least two leading bits free (zero: as far as the model force likes)
    const int rs = (int)(raw >> 63), rh = (int)(raw >> 32) ^ rs;
    int lead = clz32(rh);
    if (rh == 0) {
      const int rl = (int)raw ^ rs;
      lead = rl == 0 && rs == 0 ? 8192 : 32 + clz32(rl);
    }
    const int up = imin(lead - 2, ur - s.ud[i] - 2);
    int u;
    if constexpr (FAST) {
      raw = shl(raw, up);
      u = ur - up;
      force[i] = scaled<false>(raw - negate_if(lsr_round(s.d[i], u - s.ud[i]), sign), u);
    } else {   // the model force may be the coarser one
      const int v = ur - up;   // the common unit
      raw = shl(raw, imax(up, 0));
      u = ur - imax(up, 0);
      force[i] = scaled<true>(asr_round(raw, v - u) - negate_if(lsr_round(s.d[i], v - s.ud[i]), sign), v);
    }
    if constexpr (SUMS) {
      const int64_t m = sign ^ flip;
      z[i] = mul_signed(s.x[i], negate_if(raw, m));        // (-)|g| sign(g) raw
      uz[i] = s.ex[i] + u;
    }
  }
  if constexpr (SUMS) {
    int us = s.ew - 64;
#pragma unroll
    for (int i = 0; i < NF; ++i) us = imax(us, uz[i]);
    us += kRoom + 1;
    int64_t sum = negate_if(lsr_round(s.w - (s.w >> 2), us - (s.ew - 64)), ~(int64_t)flip);
#pragma unroll
    for (int i = 0; i < NF; ++i) sum += (asr(z[i], us - uz[i] - 1) + 1) >> 1;
    energy = from_bits(bits_of(scaled<!FAST>(sum, us)) ^ ((int64_t)flip & INT64_MIN));
  }
}

// A 1D site's share of dx^2 S (2 G + 3 V), sum_i (up_i - g_i)^2 + 3 dx^2 V, up the
// neighbour on one side (the same one at every site).  Positive terms: on a fine line
// sum_x g raw loses the gradient energy to the cancellation of its terms, 1 / |df| of
// FP64's rounding (1e-14 of the sum at 1000 sites, dx^2 = 1e-8 and fields 1e-4 about 1).
template <int NF>
CE_FX_HD double line_energy(const Fx (&g)[NF], const Fx (&up)[NF], const SiteModel<NF>& s) {
  constexpr int kRoom = NF == 1 ? 2 : (NF == 4 ? 4 : 3);   // NF squares and 3/4 w in 63 bits
  const int zw = clz64(s.w) & 63;
  const uint64_t w = s.w << zw;
  const int ew = s.ew - zw;
  uint64_t sq[NF];
  int es[NF], us = ew;
#pragma unroll
  for (int i = 0; i < NF; ++i) {
    const int e = imax(g[i].e, up[i].e);
    const int64_t d = asr(up[i].m, e - up[i].e) - asr(g[i].m, e - g[i].e);
    const uint64_t a = (uint64_t)negate_if(d, d >> 63);
    const int z = clz64(a);
    const uint64_t f = a << (z & 63);
    sq[i] = mul(f, f);
    es[i] = z == 64 ? -8192 : 2 * (e - kOne + 64 - z);
    us = imax(us, es[i]);
  }
  us += kRoom;
  int64_t sum = lsr_round(w - (w >> 2), us - ew);
#pragma unroll
  for (int i = 0; i < NF; ++i) sum += lsr_round(sq[i], us - es[i]);
  return scaled<true>(sum, us - 64);
}

}  // namespace fx
}  // namespace ce
