// ce_source.h -- how sums over the lattice enter the source 2 G + 3 V of the scale
// factor.  Plain C++: the CPU tests compile it.
#pragma once

#include <cmath>
#include <cstdint>

namespace ce {

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

}  // namespace ce
