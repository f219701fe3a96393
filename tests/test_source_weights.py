"""How the lattice sums enter a'' (`paper_0712_0813_gb300/csrc/ce_source.h`), compiled
with the host compiler (CPU; no GPU needed), and runs on boxes so large or so small that
3 dx^2 has no place in a float (GPU).

The FP64 weights are products and quotients of a few rounded numbers (4 units of 2^-53);
the pair of floats, where it is given, holds 3 dx^2 to 2^-48."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0712_0813_gb300", "csrc")

PROGRAM = r'''
#include <cstdio>
#include <initializer_list>
#include "ce_source.h"
typedef __float128 Q;

int main() {
  int bad = 0, pairs = 0, none = 0;
  for (int N = 3; N < 6200; N += 7)
    for (double L : {1e-18, 1e-12, 1e-3, 20.0, 33.3, 1e6, 1e12, 1e25, 1e100}) {
      const long long S = (long long)N * N;
      const double dx = L / N;
      const ce::SourceWeights w = ce::source_weights(dx, S);
      const Q dx2 = (Q)dx * dx, wg = 1 / (dx2 * S), wv = (Q)3 / S;
      const Q eg = (w.wg - wg) / wg, ev = (w.wv - wv) / wv, unit = (Q)0x1p-51;
      bad += eg > unit || -eg > unit || ev > unit || -ev > unit;
      if (w.ratio == w.ratio) {
        const Q er = ((Q)w.ratio + w.ratio_lo - 3 * dx2) / (3 * dx2), half = (Q)0x1p-48;
        bad += er > half || -er > half;
        ++pairs;
      } else {
        ++none;
      }
    }
  std::printf("%d %d %d\n", bad, pairs, none);
  return 0;
}
'''


def test_weights_against_quad_precision(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "w.cpp", tmp_path / "w"
    src.write_text(PROGRAM)
    r = subprocess.run([cxx, "-O2", "-std=gnu++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    if r.returncode != 0 and "float128" in r.stderr:
        pytest.skip("no quad precision in the host compiler")
    assert r.returncode == 0, r.stderr
    bad, pairs, none = (int(x) for x in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split())
    assert bad == 0
    assert pairs > 3000 and none > 1000


@pytest.mark.gpu
@pytest.mark.parametrize("kernel", ["auto", "generic", "rows", "planes"])
@pytest.mark.parametrize("precision,tol", [("f32", 2e-5), ("f64", 1e-11)])
@pytest.mark.parametrize("dims,N,L", [(3, 12, 1e25), (2, 40, 1e25), (2, 40, 1e-14), (3, 12, 20.0),
                                       (1, 100, 1e25), (1, 100, 1e160), (2, 40, 1e160), (3, 12, 1e160)])
def test_huge_and_tiny_boxes_against_the_oracle(gpu_capi, orc, dims, N, L, precision, tol, kernel):
    """Ten expanding steps: fields to the storage type's rounding (FP32: ten steps of
    2^-24 with the Laplacian's weights, 2e-5; FP64: the parity tests' 1e-11), a, a' as
    the parity tests have them (FP32 sums: 1e-5)."""
    if dims == 1 and kernel == "planes":
        pytest.skip("no such kernel in 1D")
    rng = np.random.default_rng([dims, N])
    q = (1.2,)
    f0 = 1e-2 * rng.standard_normal((2, N ** dims))
    f0[0] += 1.0
    u0 = 1e-2 * rng.standard_normal((2, N ** dims))
    dt = 0.3 * min(1.0, L / N) / dims ** 0.5
    ref = orc.init(orc.Params(dims=dims, N=N, L=L, dt=dt, nf=2, q=q, expansion=True), f0, u0)
    orc.step(ref, 10)
    with gpu_capi.Simulation(dims=dims, N=N, L=L, dt=dt, nfields=2, q=q, expansion=True, precision=precision,
                             kernel=kernel) as sim:
        sim.set_fields(f0, u0)
        sim.step(10)
        f, v, sc = sim.get_fields(gpu_capi.CE_VEL_STAGGERED)
    for got, want in ((f, ref.f), (v, ref.v)):
        got, want = got.reshape(2, -1), np.asarray(want).reshape(2, -1)
        for i in range(2):
            assert np.abs(got[i] - want[i]).max() <= tol * np.abs(want[i]).max()
    rel = 1e-5 if precision == "f32" else 1e-11
    assert sc.a == pytest.approx(ref.scale.a, rel=rel)
    assert sc.ap_half == pytest.approx(ref.scale.ap, rel=rel)
