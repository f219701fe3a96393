// ce_source.h -- the scale factor: its state, how sums over the lattice enter its
// source 2 G + 3 V, and its update.  Plain C++: the CPU tests compile it.
#pragma once

#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#define CE_HD __host__ __device__ __forceinline__
#else
#define CE_HD inline
#endif

namespace ce {

// Scale-factor state belonging to one integer time t_n.  Two slots alternate
// between step launches (launch k reads slot k%2 and writes slot (k+1)%2), so a
// launch never overwrites what its own blocks are still reading.
//
// The velocity state kept in HBM is w with  f'(t_n + dt/2) = w + c f(t_n).  The
// fused step kernel cannot add the expansion term (a''/a) f of its own kick,
// because a'' needs the global sums of the f it is writing; that term is folded
// in by the next launch through c = dt a''/a (and c = 0 after a restore).
struct DevScalars {
  double a;    // a(t_n)
  double ap;   // a'(t_n + dt/2)
  double app;  // a''(t_n)
  double s;    // a''(t_n) / a(t_n)
  double c;    // coefficient of f in the velocity reconstruction above
};

// 2 G + 3 V = wg sum of (df)^2 + wv sum of V = wg (sum of (df)^2 + ratio sum of V).
// FP64 sums take the two weights.  FP32 sums, which are added as float pairs, take
// ratio = 3 dx^2 as such a pair; it is NaN where a pair does not hold it (or its
// products' residuals) to 2^-48, and those blocks then take the FP64 weights.
struct SourceWeights {
  double wg, wv;
  float ratio, ratio_lo;
};

inline SourceWeights source_weights(double dx, int64_t S) {
  SourceWeights w;
  w.wg = 1.0 / (dx * dx * (double)S);
  w.wv = 3.0 / (double)S;
  const double ratio = 3.0 * dx * dx;
  const bool pair = ratio >= 0x1p-90 && ratio <= 0x1p90;
  w.ratio = pair ? (float)ratio : NAN;
  w.ratio_lo = pair ? (float)(ratio - (double)w.ratio) : 0.f;
  return w;
}

// Scale-factor update of reading c-4, done once per step by one thread:
//   a_{n+1} = a_n + dt a'_{n+1/2}
//   Q = kappa2 (2 G + 3 V) / a_{n+1},  C = 2 a'_{n+1/2} + dt Q
//   u = a'_{n+3/2} + a'_{n+1/2} = 2 C / (1 + sqrt(1 + dt C / a_{n+1}))
// (closed form of the implicit midpoint a'_new - a'_old = dt (-(u/2)^2/a + Q)),
//   a''_{n+1} = (u - 2 a'_{n+1/2}) / dt,  a'_{n+3/2} = u - a'_{n+1/2}.
// In two parts: what does not need the sums (scale_ahead) can run before they are
// there.  y = u / C solves (e/4) y^2 + y = 1 with e = dt C / a: for small e two
// Newton steps in FP64 with FP32's slope, from FP32's root (errors 1e-7, 1e-14, 0),
// are six instructions where the square root and the division take eighteen.
// Products that meet a sum are written as FMAs: left to the compiler, copies of this
// code in one kernel rounded differently, and a run's bits depended on how its steps
// were shared out to calls.
struct ScaleAhead {
  double a, ap, ap2, ia, dia, k1, e1;
};
CE_HD ScaleAhead scale_ahead(const DevScalars& in, double dt, double kappa2) {
  ScaleAhead s;
  s.a = fma(dt, in.ap, in.a);
  s.ap = in.ap;
  s.ap2 = in.ap + in.ap;
  s.ia = 1.0 / s.a;
  s.dia = dt * s.ia;
  s.k1 = kappa2 * s.dia;
  s.e1 = 0.25 * s.dia;
  return s;
}
// source: 2 G + 3 V.  False where there is no real a', or the source is not finite.
CE_HD bool scale_update(const ScaleAhead& s, DevScalars& out, double source, double inv_dt) {
  const double C = fma(s.k1, source, s.ap2);
  const double e4 = s.e1 * C;
  const float e = 4.f * (float)e4;
  bool ok = true;
  double y;
  if (fabsf(e) < 0.25f) {
    const float yf = 2.f / (1.f + sqrtf(1.f + e));
    const double slope = (double)(1.f / fmaf(0.5f * e, yf, 1.f));
    y = (double)yf;
    y = fma(fma(-(e4 * y), y, 1.0 - y), slope, y);
    y = fma(fma(-(e4 * y), y, 1.0 - y), slope, y);
  } else {   // also where something is not finite
    const double disc = fma(4.0, e4, 1.0);
    ok = disc >= 0.0 && fabs(source) <= 1.7976931348623157e308;
    y = 2.0 / (1.0 + sqrt(disc));
  }
  const double app = fma(C, y, -s.ap2) * inv_dt;
  out.c = app * s.dia;
  out.app = app;
  out.s = app * s.ia;
  out.a = s.a;
  out.ap = fma(C, y, -s.ap);
  return ok;
}

}  // namespace ce
