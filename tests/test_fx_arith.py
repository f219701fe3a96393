"""The integer arithmetic of the FP64 step's force
(`paper_0712_0813_gb300/csrc/ce_fx.cuh`), compiled with the host compiler and
compared with quad precision (CPU; no GPU needed):

* every double converts to the integer form and back bit for bit, and scaled
  integers convert to the nearest double;
* the force of a site over random stencils -- smooth, rough, of any sign, with a
  zero field, with exponents spread over 80 binary orders, with dx^2 V'' from 1e-8
  to 1000 (the fast and the general form), near the range's ends -- is within
  2^-53 |force| (its one rounding) + (2d + 2) 2^-57 of the stencil's largest value
  (what alignment drops of the 2d + 1 words of the Laplacian, and half a unit of the
  aligned model force, a unit being at most 2^-57 of that value) + 2^-56 of the
  model force (its products keep 58 bits and more), and its largest error is no
  larger than FP64's on the same stencils;
* the energy term, the sum over the fields of g times such a sum, is within 2^-53 of
  itself + the same errors times |g| + one unit a field for the product (a unit of
  it is at most 2^-56 of |g| times the stencil's largest value) + (nf + 1) half
  units of the common grid, up to eight times as coarse as the coarsest of those
  units and of 4 dx^2 V's (at most 2^-57 of it, and four of them for its products);
  and its mean error, which the sum over a lattice would carry, is within 2^-56 of
  its terms' sizes (what rounding 4 dx^2 V's products down adds on average).

The program prints each largest error over its bound."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0712_0813_gb300", "csrc")

PROGRAM = r'''
#include <cmath>
#include <cstdio>
#include <random>
#include "ce_fx.cuh"
using namespace ce::fx;
typedef __float128 Q;

FxConst constant(long double v) {
  FxConst c{0, -4096};
  if (!(v > 0)) return c;
  int e;
  c.m = (uint64_t)std::ldexp(std::frexp(v, &e), 64);
  c.e = e;
  return c;
}

template <int NF, int D>
void run(const char* name, double base, double amp, double dx2, double q0, bool wild) {
  std::mt19937_64 r(NF * 100 + D);
  std::normal_distribution<double> n(0, 1);
  std::uniform_int_distribution<int> U(-40, 40);
  const double q[3] = {q0, 5.0, 40.0};
  FxModel k;
  k.dx2 = constant(dx2);
  for (int i = 0; i < 3; ++i) {
    k.q[i] = constant(q[i]);
    k.qdx2[i] = constant((long double)q[i] * dx2);
  }
  double force = 0, worst = 0, worst64 = 0, energy = 0, bias = 0;
  long fast = 0, terms = 0;
  const int sites = 60000;
  for (int it = 0; it < sites; ++it) {
    double g[NF], nb[NF][2 * D];
    Fx G[NF], NB[NF][2 * D];
    const bool zero = it % 97 == 5;
    for (int i = 0; i < NF; ++i)
      for (int j = -1; j < 2 * D; ++j) {
        double v = (i == 0 ? base : 0.0) + amp * n(r);
        if (wild) v = std::ldexp(n(r), U(r));
        if (zero && i == NF - 1 && NF > 1) v = 0.0;
        (j < 0 ? g[i] : nb[i][j]) = v;
        (j < 0 ? G[i] : NB[i][j]) = from_double(v);
      }
    int em[NF];
    SiteModel<NF> s;
    double F[NF], en;
    stencil_exponents<NF, D>(G, NB, em);
    site_model<NF, true>(G, k, s);
    if (fast_site<NF>(em, s)) {
      ++fast;
      site_force<NF, D, true, true>(G, NB, em, s, -(it & 1), F, en);
    } else {
      site_force<NF, D, true, false>(G, NB, em, s, -(it & 1), F, en);
    }
    Q cpl = 0, eq = 0;
    double cd = 0, mag = 0, slack = 0, grid = 0, pot = 0;
    for (int i = 1; i < NF; ++i) {
      cpl += (Q)q[i - 1] * g[i] * g[i];
      cd = std::fma(q[i - 1] * g[i], g[i], cd);
    }
    for (int i = 0; i < NF; ++i) {
      Q raw = -2 * D * (Q)g[i];
      double sum = 0, mx = std::fabs(g[i]), size = 2 * D * mx;
      for (int j = 0; j < 2 * D; ++j) {
        raw += nb[i][j];
        sum += nb[i][j];
        size += std::fabs(nb[i][j]);
        mx = std::fmax(mx, std::fabs(nb[i][j]));
      }
      const Q dv = i == 0 ? (Q)g[0] * ((Q)g[0] * g[0] + cpl) : (Q)q[i - 1] * g[0] * g[0] * g[i];
      const double dvd = i == 0 ? g[0] * std::fma(g[0], g[0], cd) : q[i - 1] * (g[0] * g[0]) * g[i];
      const Q f = raw - (Q)dx2 * dv;
      const double f64 = std::fma(-dx2, dvd, std::fma(-2.0 * D, g[i], sum));
      const double model = std::fabs((double)((Q)dx2 * dv));
      size += model;
      slack += std::fabs(g[i]) * (std::ldexp((2 * D + 4) * mx, -57) + std::ldexp(model, -56));
      pot += std::fabs(g[i]) * model;
      grid = std::fmax(grid, std::fabs(g[i]) * mx);
      if (size > 0) {
        const double bound =
            std::ldexp(std::fabs((double)f), -53) + std::ldexp((2 * D + 2) * mx, -57) + std::ldexp(model, -56);
        force = std::fmax(force, std::fabs((double)(F[i] - f)) / bound);
        worst = std::fmax(worst, std::fabs((double)(F[i] - f)) / size);
        worst64 = std::fmax(worst64, std::fabs((double)(f64 - f)) / size);
      } else if (F[i] != 0.0) {
        force = 1e9;
      }
      eq += (Q)g[i] * (raw - (Q)0.75 * (Q)dx2 * dv);
      mag += std::fabs(g[i]) * size;
    }
    if (mag > 0) {
      const double e = (double)((Q)en - eq);
      energy = std::fmax(energy, std::fabs(e) / (std::ldexp(std::fabs((double)eq), -53) + slack +
                                                 std::ldexp((NF + 1) * grid, -54) + std::ldexp((NF + 2) * pot, -55)));
      bias += e / std::ldexp(mag, -56);
      ++terms;
    }
  }
  std::printf("%s_nf%d_%dd %.6f %.6f %.6f %.6f %.4f\n", name, NF, D, force, worst / worst64, energy, bias / terms,
              (double)fast / sites);
}

int main() {
  const double v[] = {0.0, -0.0, 1.0, -1.5, 5e-324, -5e-324, 2.2250738585072014e-308, -2.2e-308, 1.7976931348623157e308,
                      INFINITY, -INFINITY, 3.14159, -1e-300};
  int bad = 0;
  for (double x : v) bad += bits_of(to_double(from_double(x))) != bits_of(x) && x != 0.0;
  std::mt19937_64 r(7);
  for (int i = 0; i < 200000; ++i) {
    const int64_t m = (int64_t)r() >> (1 + r() % 62);
    const int u = (int)(r() % 400) - 200;
    const double want = (double)std::ldexp((long double)m, u);
    // halves round upwards in size: at most one unit from the nearest-even double
    const double got = scaled<true>(m, u);
    bad += !(std::fabs((double)((Q)got - std::ldexp((long double)m, u))) <= std::ldexp(std::fabs(want), -53));
    bad += scaled<false>(m, u) != got;
  }
  std::printf("conversions_nf0_0d %d 0 0 0 0\n", bad);
  run<2, 3>("smooth", 1.0, 1e-2, 0.0061, 1.2, false);
  run<2, 3>("coarse", 1.0, 1e-4, 0.39, 1.2, false);
  run<1, 3>("smooth", 1.0, 1e-2, 0.0061, 1.2, false);
  run<4, 3>("rough", 1.0, 0.1, 0.0061, 0.8, false);
  run<2, 2>("strong", 2.0, 1e-2, 1e-5, 200.0, false);
  run<3, 3>("massive", 3.0, 1.0, 40.0, 200.0, false);
  run<2, 1>("fine", 1.0, 1e-2, 1e-8, 1.2, false);
  run<2, 3>("negative", -1.0, 1e-2, 0.0061, 1.2, false);
  run<2, 3>("wild", 1.0, 1.0, 0.01, 1.2, true);
  run<4, 2>("wild", 1.0, 1.0, 1e-3, 1.2, true);
  run<2, 3>("large", 1e60, 1e58, 0.0061, 1.2, false);
  run<2, 3>("small", 1e-90, 1e-92, 0.0061, 1.2, false);
  return 0;
}
'''


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("fx")
    src, exe = os.path.join(d, "fx.cpp"), os.path.join(d, "fx")
    with open(src, "w") as f:
        f.write(PROGRAM)
    r = subprocess.run([cxx, "-O2", "-std=gnu++17", "-ffp-contract=off", "-I", CSRC, src, "-o", exe],
                       capture_output=True, text=True)
    if r.returncode != 0 and "float128" in r.stderr:
        pytest.skip("no quad precision in the host compiler")
    assert r.returncode == 0, r.stderr
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    return {line.split()[0]: [float(x) for x in line.split()[1:]] for line in out.splitlines()}


def test_conversions(errors):
    assert errors["conversions_nf0_0d"][0] == 0


def test_force_and_energy_against_quad_precision(errors):
    cases = {k: v for k, v in errors.items() if not k.startswith("conversions")}
    assert len(cases) == 12
    for name, (force, against_fp64, energy, bias, fast) in cases.items():
        assert force <= 1.0, (name, force)
        assert against_fp64 <= 1.0, (name, against_fp64)
        assert energy <= 1.0 and abs(bias) <= 1.0, (name, energy, bias)
    assert cases["smooth_nf2_3d"][4] == 1.0 and cases["massive_nf3_3d"][4] == 0.0
    assert 0.0 < cases["wild_nf2_3d"][4] < 1.0
