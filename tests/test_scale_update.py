"""The scale-factor update (`paper_0712_0813_gb300/csrc/ce_source.h`) against quad
precision (CPU; no GPU needed).

* One update: u = a'_{n+3/2} + a'_{n+1/2} within 8 units of 2^-53 (the chain a, 1/a,
  dt/a, C, e, two Newton steps, u has eight roundings), for small e by the Newton
  steps, beyond by the square root; a' = u - a'_{n+1/2} to 12 of them, in units of
  |u| + |a'|; a'' = (u - 2 a') / dt likewise over dt.
* Runs of 1000 steps with a source that falls and oscillates as that of the lattice
  does: a and a' end, over 600 runs, no further from the exact recurrence than with the
  closed form evaluated by FP64's own square root and division, operation by operation
  (mean and largest error)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0712_0813_gb300", "csrc")

PROGRAM = r'''
#include <cstdio>
#include <cmath>
#include <initializer_list>
#include <random>
#include "ce_source.h"
typedef __float128 Q;
using namespace ce;

Q root(Q x) {   // Newton from FP64's root
  Q r = std::sqrt((double)x);
  for (int k = 0; k < 3; ++k) r = (r + x / r) / 2;
  return r;
}
double size(Q x) { return std::fabs((double)x); }

template <typename T>
struct Plain {   // the closed form, operation by operation
  T a, ap, u;
  template <typename Root>
  void step(T source, T dt, T kappa2, Root rt) {
    a = a + dt * ap;
    const T C = T(2) * ap + dt * (kappa2 * source / a);
    u = T(2) * C / (T(1) + rt(T(1) + dt * C / a));
    ap = u - ap;
  }
};

int main() {
  const double kappa2 = 8.0 * M_PI / 3.0 * 0.342 * 0.342;
  std::mt19937_64 r(5);
  std::uniform_real_distribution<double> U(0.0, 1.0);
  double one = 0, oneap = 0, oneapp = 0;
  int large = 0;
  for (int it = 0; it < 200000; ++it) {
    const double dt = std::exp(-9.0 + 9.0 * U(r)), a = std::exp(3.0 * U(r));
    const double ap = (2.0 * U(r) - 0.5) * (it % 3 ? 1.0 : 0.01), source = it % 5 ? U(r) : 50.0 * U(r);
    DevScalars in{a, ap, 0, 0, 0}, out;
    const bool ok = scale_update(scale_ahead(in, dt, kappa2), out, source, 1.0 / dt);
    const Q qa = (Q)a + (Q)dt * ap, C = 2 * (Q)ap + (Q)dt * kappa2 * source / qa, disc = 1 + (Q)dt * C / qa;
    if (disc < 0) {
      if (ok) one = 1e9;
      continue;
    }
    if (!ok) one = 1e9;
    large += std::fabs((double)(disc - 1)) >= 0.25;
    const Q u = 2 * C / (1 + root(disc));
    // C is a sum of two terms: its roundings are units of them
    const double terms = 2 * std::fabs(ap) + dt * kappa2 * source / (double)qa, unit = std::ldexp(terms, -53);
    one = std::fmax(one, size((Q)out.ap + ap - u) / (8 * unit));
    oneap = std::fmax(oneap, size((Q)out.ap - (u - ap)) / (12 * unit));
    oneapp = std::fmax(oneapp, size((Q)out.app - (u - 2 * (Q)ap) / dt) * dt / (12 * unit));
  }
  std::printf("one %.4f %.4f %.4f %d\n", one, oneap, oneapp, large);
  double mean[4] = {0, 0, 0, 0}, worst[4] = {0, 0, 0, 0};
  for (double dt : {0.05, 0.02, 0.004})
    for (int run = 0; run < 200; ++run) {
      const double s0 = 0.8 + 0.4 * U(r), w = 1.0 + 2.0 * U(r), ap0 = std::sqrt(kappa2 * 0.25 * s0);
      DevScalars now{1.0, ap0, 0, 0, 0}, next;
      Plain<double> d{1.0, ap0, 0};
      Plain<Q> q{1, ap0, 0};
      for (int k = 0; k < 1000; ++k) {
        const double t = k * dt, source = s0 * (0.6 + 0.4 * std::cos(w * t)) / (1.0 + 0.02 * t);
        scale_update(scale_ahead(now, dt, kappa2), next, source, 1.0 / dt);
        now = next;
        d.step(source, dt, kappa2, [](double x) { return std::sqrt(x); });
        q.step(source, dt, kappa2, root);
      }
      const double e[4] = {size((now.a - q.a) / q.a), size((d.a - q.a) / q.a), size((now.ap - q.ap) / q.ap),
                           size((d.ap - q.ap) / q.ap)};
      for (int j = 0; j < 4; ++j) {
        mean[j] += e[j] / 600;
        worst[j] = std::fmax(worst[j], e[j]);
      }
    }
  std::printf("a %.3g %.3g %.3g %.3g\n", mean[0], mean[1], worst[0], worst[1]);
  std::printf("ap %.3g %.3g %.3g %.3g\n", mean[2], mean[3], worst[2], worst[3]);
  return 0;
}
'''


def test_scale_update_against_quad_precision(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "scale.cpp", tmp_path / "scale"
    src.write_text(PROGRAM)
    r = subprocess.run([cxx, "-O2", "-std=gnu++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    if r.returncode != 0 and "float128" in r.stderr:
        pytest.skip("no quad precision in the host compiler")
    assert r.returncode == 0, r.stderr
    out = {line.split()[0]: [float(x) for x in line.split()[1:]]
           for line in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines()}
    u, ap, app, large = out["one"]
    assert u <= 1.0 and ap <= 1.0 and app <= 1.0 and large > 1000
    for name in ("a", "ap"):
        mean, mean_plain, worst, worst_plain = out[name]
        assert mean <= mean_plain and worst <= worst_plain, (name, out[name])
