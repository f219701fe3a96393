// ce_fx_force.cuh -- the force of a site by the form its values allow: the fast or
// the general integer form of ce_fx.cuh, or FP64 where a value is not finite.
#pragma once

#include "ce_device.cuh"
#include "ce_fx.cuh"

namespace ce {
namespace fx {

// The force of a site one of whose stencil values is infinite or NaN, in FP64.
template <int NF, int DIMS>
static __device__ __noinline__ void force_fp64(const double* g, const double* nb, double dx2, const double* q, double* force,
                                        double* energy) {
  double gs[NF], dv[NF], vs, e = 0.0;
  for (int i = 0; i < NF; ++i) gs[i] = g[i];
  const double qs[3] = {q[0], q[1], q[2]};
  model_dv<double, NF>(gs, qs, dv, vs);
  for (int i = 0; i < NF; ++i) {
    double raw = -2.0 * DIMS * gs[i];
    for (int j = 0; j < 2 * DIMS; ++j) raw += nb[i * 2 * DIMS + j];
    force[i] = fma(-dx2, dv[i], raw);
    if constexpr (DIMS == 1) {
      const double df = nb[i * 2 + 1] - gs[i];
      e -= df * df;
    } else {
      e += gs[i] * fma(-0.75 * dx2, dv[i], raw);
    }
  }
  *energy = DIMS == 1 ? fma(-3.0 * dx2, vs, e) : e;
}

// The site's force by the form its values allow; GENERAL leaves the fast form out, for
// kernels whose code is long enough without it.  In 1D the energy term is that of
// line_energy, with its sign turned.
template <int NF, int DIMS, bool SUMS, bool GENERAL = false>
__device__ __forceinline__ void force_of(const Fx (&g)[NF], const Fx (&nb)[NF][2 * DIMS], const FxModel& k,
                                         double inv_dx2, const double (&q)[3], double (&force)[NF], double& energy) {
  const int flip = -(int)(threadIdx.x & 1u);
  int em[NF];
  stencil_exponents<NF, DIMS>(g, nb, em);
  SiteModel<NF> s;
  site_model<NF, SUMS>(g, k, s);
  Fx up[NF];
#pragma unroll
  for (int i = 0; i < NF; ++i) up[i] = nb[i][1];
  constexpr bool kParts = SUMS && DIMS > 1;
  if (!GENERAL && fast_site<NF>(em, s)) {
    site_force<NF, DIMS, kParts, true>(g, nb, em, s, flip, force, energy);
    if constexpr (SUMS && DIMS == 1) energy = -line_energy<NF>(g, up, s);
    return;
  }
  int most = em[0];
#pragma unroll
  for (int i = 1; i < NF; ++i) most = max(most, em[i]);
  if (most < kNonFinite) {
    site_force<NF, DIMS, kParts, false>(g, nb, em, s, flip, force, energy);
    if constexpr (SUMS && DIMS == 1) energy = -line_energy<NF>(g, up, s);
    return;
  }
  double gd[NF], nd[NF * 2 * DIMS], fd[NF], qd[3] = {q[0], q[1], q[2]}, ed;
#pragma unroll
  for (int i = 0; i < NF; ++i) {
    gd[i] = to_double(g[i]);
#pragma unroll
    for (int j = 0; j < 2 * DIMS; ++j) nd[i * 2 * DIMS + j] = to_double(nb[i][j]);
  }
  force_fp64<NF, DIMS>(gd, nd, 1.0 / inv_dx2, qd, fd, &ed);
#pragma unroll
  for (int i = 0; i < NF; ++i) force[i] = fd[i];
  energy = ed;
}

}  // namespace fx
}  // namespace ce
