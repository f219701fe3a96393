"""Energies of FP32 lattices against FP64 sums of the same FP32 site terms.

The site terms are formed here in FP32 as the library forms them (an FMA as a product and
sum in FP64, rounded once to FP32: off by one unit, 2^-24 of the site, on rare ties) and
added in FP64.  The library's pairs of floats hold 2^-40 of a sum and better; 5e-11 leaves
room for 2^-24 at 50 of 65536 sites.  Plain FP32 sums of 16 sites were off by 1e-9 to
1.5e-8 here."""
import numpy as np
import pytest

from paper_0712_0813_gb300.icgen import courant_dt

pytestmark = pytest.mark.gpu

f32 = np.float32


def fma(a, b, c):
    return (a.astype(np.float64) * b + np.asarray(c, dtype=np.float64)).astype(f32)


@pytest.mark.parametrize("dims,N,nf", [(1, 65536, 2), (2, 301, 4), (3, 64, 2), (3, 41, 3), (3, 101, 1), (2, 1200, 2)])
def test_energies_are_fp64_sums_of_the_site_terms(gpu_capi, dims, N, nf):
    L, q = 20.0, (0.8, 5.0, 40.0)[:nf - 1]
    rng = np.random.default_rng([dims, N, nf])
    f0 = 1e-2 * rng.standard_normal((nf, N ** dims))
    f0[0] += 1.0
    with gpu_capi.Simulation(dims=dims, N=N, L=L, dt=courant_dt(dims, N, L, 1.0, q), nfields=nf, q=q, expansion=True,
                             precision="f32") as sim:
        sim.set_fields(f0, np.zeros_like(f0))
        sim.step(2)
        e = sim.energy()
        f = sim.get_fields(gpu_capi.CE_VEL_STAGGERED)[0].astype(f32).reshape((nf,) + (N,) * dims)
    for i in range(nf):
        g2 = np.zeros_like(f[i])
        for d in range(dims):
            df = np.roll(f[i], -1, dims - 1 - d) - f[i]
            g2 = fma(df, df, g2)
        assert e["G"][i] == pytest.approx(0.5 * (N / L) ** 2 * g2.astype(np.float64).mean(), rel=5e-11)
    phi2 = f[0] * f[0]
    cpl = np.zeros_like(phi2)
    for qi, x in zip(q, f[1:]):
        cpl = fma(f32(qi) * x, x, cpl)
    v = phi2 * fma(np.full_like(phi2, 0.25), phi2, f32(0.5) * cpl)
    assert e["V"] == pytest.approx(v.astype(np.float64).mean(), rel=5e-11)
