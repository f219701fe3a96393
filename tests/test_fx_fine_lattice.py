"""The FP64 step's integer force (`paper_0712_0813_gb300/csrc/ce_fx.cuh`) where the
Laplacian is far below the fields it is formed of -- homogeneous lattices, fields a
few units in the last place from one, fine spacings -- compared with quad precision
(CPU; no GPU needed).

All values of a stencil lie within a binade or two here, so nothing is lost in
aligning them and raw, the sum over the neighbours, is exact.  Bounds, M standing for
dx^2 |dV/df| and e for the energy term:

* force: 2^-53 |force| (its rounding to a double) + 2^-54 M + 2^-62 |raw|.  The
  products of M keep 58 bits (2^-56 M); M and raw meet in a unit of at most four of
  M's own, of which M has at least 2^57, and each is rounded there once (2 x 2^-56 M),
  or in a unit of raw's own, of which raw has at least 2^61 (half of one, for M);
* energy term: 2^-53 |e| + 2^-51 sum |g| M + 2^-55 sum |g raw|: 4 dx^2 V has at least
  2^56 units and the common grid at most eight of them, in which up to five terms are
  rounded to half a unit; a product with raw keeps 60 bits of it, or a unit of M's.

A force formed in a unit of the fields themselves misses these by a factor that grows
with 1 / dx^2: 10 at dx^2 = 0.006, 10^9 at 10^-10."""
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

double size(Q x) { return std::fabs((double)x); }

// Fields of random size and sign; each neighbour within `ulps` units of the site.
template <int NF, int D>
void run(double dx2, int ulps) {
  std::mt19937_64 r(NF * 100 + D + ulps);
  std::uniform_real_distribution<double> U(0.25, 2.0);
  std::uniform_int_distribution<int> W(-ulps, ulps);
  const double q[3] = {1.2, 5.0, 40.0};
  FxModel k;
  k.dx2 = constant(dx2);
  for (int i = 0; i < 3; ++i) {
    k.q[i] = constant(q[i]);
    k.qdx2[i] = constant((long double)q[i] * dx2);
  }
  double force = 0, energy = 0;
  for (int it = 0; it < 20000; ++it) {
    double g[NF], nb[NF][2 * D];
    Fx G[NF], NB[NF][2 * D];
    for (int i = 0; i < NF; ++i) {
      g[i] = (r() & 1 ? 1 : -1) * U(r);
      G[i] = from_double(g[i]);
      for (int j = 0; j < 2 * D; ++j) {
        nb[i][j] = g[i] + W(r) * 0x1p-52;
        NB[i][j] = from_double(nb[i][j]);
      }
    }
    int em[NF];
    SiteModel<NF> s;
    double F[NF], en;
    stencil_exponents<NF, D>(G, NB, em);
    site_model<NF, true>(G, k, s);
    if (fast_site<NF>(em, s)) site_force<NF, D, true, true>(G, NB, em, s, -(it & 1), F, en);
    else site_force<NF, D, true, false>(G, NB, em, s, -(it & 1), F, en);
    Q cpl = 0, e = 0;
    double pot = 0, grad = 0;
    for (int i = 1; i < NF; ++i) cpl += (Q)q[i - 1] * g[i] * g[i];
    for (int i = 0; i < NF; ++i) {
      Q raw = -2 * D * (Q)g[i];
      for (int j = 0; j < 2 * D; ++j) raw += nb[i][j];
      const Q m = (Q)dx2 * (i == 0 ? (Q)g[0] * ((Q)g[0] * g[0] + cpl) : (Q)q[i - 1] * g[0] * g[0] * g[i]);
      const Q f = raw - m;
      force = std::fmax(force, size(F[i] - f) / (std::ldexp(size(f), -53) + std::ldexp(size(m), -54) + std::ldexp(size(raw), -62)));
      e += (Q)g[i] * (raw - (Q)0.75 * m);
      pot += size((Q)g[i] * m);
      grad += size((Q)g[i] * raw);
    }
    energy = std::fmax(energy, size(en - e) / (std::ldexp(size(e), -53) + std::ldexp(pot, -51) + std::ldexp(grad, -55)));
  }
  std::printf("nf%d_%dd_dx2_%g_ulps%d %.4f %.4f\n", NF, D, dx2, ulps, force, energy);
}

template <int NF, int D>
void spacings() {
  for (double dx2 : {10.0, 0.39, 0.0061, 1.6e-6, 9.3e-8, 1e-12, 1e-20})
    for (int ulps : {0, 3, 4000}) run<NF, D>(dx2, ulps);
}

int main() {
  spacings<1, 1>();
  spacings<2, 1>();
  spacings<4, 1>();
  spacings<1, 2>();
  spacings<2, 2>();
  spacings<2, 3>();
  spacings<3, 3>();
  spacings<4, 3>();
  return 0;
}
'''


def test_fine_lattices_against_quad_precision(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "fine.cpp", tmp_path / "fine"
    src.write_text(PROGRAM)
    r = subprocess.run([cxx, "-O2", "-std=gnu++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    if r.returncode != 0 and "float128" in r.stderr:
        pytest.skip("no quad precision in the host compiler")
    assert r.returncode == 0, r.stderr
    lines = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines()
    assert len(lines) == 8 * 7 * 3
    for name, force, energy in (x.split() for x in lines):
        assert float(force) <= 1.0 and float(energy) <= 1.0, (name, force, energy)
