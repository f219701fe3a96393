"""The integer force of the FP64 step (`paper_0712_0813_gb300/csrc/ce_fx.cuh`) below
FP64's normal range (CPU; no GPU needed): scaled integers convert to the nearest
subnormal (ties may go either way: at most half a unit of 2^-1074), and the force of a
stencil of tiny values is the sum over its neighbours, which FP64 forms exactly there."""
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

int main() {
  std::mt19937_64 r(11);
  int bad = 0, forces = 0, nonzero = 0;
  for (int it = 0; it < 200000; ++it) {
    const int64_t m = (int64_t)r() >> (1 + r() % 62);
    const int u = -1150 + (int)(r() % 120);
    Q exact = m;   // the range of quad precision holds m 2^u
    for (int k = 0; k < -u; ++k) exact /= 2;
    const double got = scaled<true>(m, u);
    const Q err = (Q)got - exact, half = (Q)5e-324 / 2;
    const Q rel = (exact < 0 ? -exact : exact) / (Q)9007199254740992.0;   // 2^-53 of it
    const Q bound = half > rel ? half : rel;
    bad += err > bound || -err > bound || scaled<false>(m, u) != got;
  }
  FxModel k{{0x8000000000000000ull, -4}, {{0x8000000000000000ull, 1}}, {{0x8000000000000000ull, -3}}};
  for (int it = 0; it < 200000; ++it) {
    const int bits = 1 + r() % 56;   // of a value in units of 2^-1074
    double g[2], nb[2][6];
    Fx G[2], NB[2][6];
    for (int i = 0; i < 2; ++i)
      for (int j = -1; j < 6; ++j) {
        const double v = (r() & 1 ? 1 : -1) * (double)(r() >> (64 - bits)) * 5e-324;
        (j < 0 ? g[i] : nb[i][j]) = v;
        (j < 0 ? G[i] : NB[i][j]) = from_double(v);
      }
    int em[2];
    SiteModel<2> s;
    double F[2], en;
    stencil_exponents<2, 3>(G, NB, em);
    site_model<2, true>(G, k, s);
    if (fast_site<2>(em, s)) site_force<2, 3, true, true>(G, NB, em, s, 0, F, en);
    else site_force<2, 3, true, false>(G, NB, em, s, 0, F, en);
    for (int i = 0; i < 2; ++i) {
      Q raw = -6 * (Q)g[i];
      for (int j = 0; j < 6; ++j) raw += nb[i][j];
      const Q err = (Q)F[i] - raw, rel = (raw < 0 ? -raw : raw) / (Q)9007199254740992.0;
      forces += err > rel || -err > rel;   // exact up to 53 bits, then rounded
      nonzero += F[i] != 0.0;
    }
  }
  std::printf("%d %d %d\n", bad, forces, nonzero);
  return 0;
}
'''


def test_subnormal_results(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "sub.cpp", tmp_path / "sub"
    src.write_text(PROGRAM)
    r = subprocess.run([cxx, "-O2", "-std=gnu++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    if r.returncode != 0 and "float128" in r.stderr:
        pytest.skip("no quad precision in the host compiler")
    assert r.returncode == 0, r.stderr
    bad, forces, nonzero = (int(x) for x in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split())
    assert bad == 0 and forces == 0
    assert nonzero > 300000
