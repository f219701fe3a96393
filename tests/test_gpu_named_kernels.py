"""Kernels named by the caller, on shapes where the automatic choice takes another one:
the FP64 kernels that take one launch a step and the FP32 column kernel at the sides
where strips and row groups end raggedly."""
import numpy as np
import pytest

from paper_0712_0813_gb300.icgen import courant_dt, lattice_ics
from test_gpu_parity import CASES, TOL64, per_field_err, relmax, run_pair

pytestmark = pytest.mark.gpu

Q = (0.8, 5.0, 40.0)
# 2D with 1, 3 and 4 fields: every neighbour wraps (3), one-site last strips (31, 61),
# ragged ones (37, 101), several chunks of rows (257)
SQUARES = [(2, N, 20.0, 0.9 * courant_dt(2, N, 20.0, 1.0, Q[:nf - 1]), nf, Q[:nf - 1], expansion)
           for N, nf, expansion in ((3, 3, True), (31, 1, True), (37, 4, True), (61, 3, False), (101, 3, True),
                                    (257, 4, True), (257, 1, False))]


@pytest.mark.parametrize("case", CASES + SQUARES,
                         ids=[f"{c[0]}d_N{c[1]}_nf{c[4]}_{'exp' if c[6] else 'flat'}" for c in CASES + SQUARES])
def test_fp64_generic_kernel_100_steps_against_the_oracle(gpu_capi, orc, case):
    """The parity tests' bound, on kernel="generic"."""
    dims, N, L, dt, nf, q, expansion = case
    ref, sim, f, v, sc = run_pair(orc, gpu_capi, dims, N, L, dt, nf, q, expansion, 100, kernel="generic")
    with sim:
        assert sim.kernel == gpu_capi.CE_KERNEL_GENERIC
        assert per_field_err(f, ref.f, nf) <= TOL64
        assert per_field_err(v, ref.v, nf) <= TOL64
        assert sc.step == 100 and sc.t == ref.scale.t
        if expansion:
            assert abs(sc.a - ref.scale.a) / ref.scale.a <= TOL64
            assert abs(sc.ap_half - ref.scale.ap) / abs(ref.scale.ap) <= TOL64
            assert abs(sc.app - ref.scale.app) / abs(ref.scale.app) <= 1e-9


@pytest.mark.parametrize("nf", [1, 2, 4])
@pytest.mark.parametrize("N", [3, 33, 37, 61, 101])
def test_fp32_column_kernel_fields_equal_generic(gpu_capi, N, nf):
    """Without expansion the two kernels do the same operations at a site."""
    q = Q[:nf - 1]
    f0, u0 = lattice_ics(3, N, 20.0, nf, q=q, seed=4, amp=1e-2)
    out = []
    for kernel in ("planes", "generic"):
        with gpu_capi.Simulation(dims=3, N=N, L=20.0, dt=0.02, nfields=nf, q=q, expansion=False, precision="f32",
                                 kernel=kernel) as sim:
            sim.set_fields(f0, u0)
            sim.step(20)
            out.append(sim.get_fields(gpu_capi.CE_VEL_STAGGERED))
    (fa, va, _), (fb, vb, _) = out
    assert np.array_equal(fa, fb) and np.array_equal(va, vb)


@pytest.mark.parametrize("kernel", ["auto", "generic"])
@pytest.mark.parametrize("expansion", [True, False])
@pytest.mark.parametrize("dims,N,L", [(1, 4096, 0.2), (2, 64, 0.01), (3, 16, 1e-4)])
def test_fp64_homogeneous_fields_on_a_fine_lattice(gpu_capi, orc, dims, N, L, expansion, kernel):
    """The Laplacian is exactly zero, so the model force alone moves the fields: 100
    steps to 1e-12 of fields and velocities (rounding: 100 x 2^-53), alike at every
    site.  A force in a unit of the fields was off by 1e-9 and more here."""
    q = (1.2,)
    f0 = np.empty((2, N ** dims))
    f0[0], f0[1] = 0.9, 0.3
    u0 = np.zeros_like(f0)
    dt = courant_dt(dims, N, L, 1.0, q)
    ref = orc.init(orc.Params(dims=dims, N=N, L=L, dt=dt, nf=2, q=q, expansion=expansion), f0, u0)
    orc.step(ref, 100)
    with gpu_capi.Simulation(dims=dims, N=N, L=L, dt=dt, nfields=2, q=q, expansion=expansion, kernel=kernel) as sim:
        sim.set_fields(f0, u0)
        sim.step(100)
        f, v, sc = sim.get_fields(gpu_capi.CE_VEL_STAGGERED)
    for got, want in ((f, ref.f), (v, ref.v)):
        for g, w in zip(got.reshape(2, -1), np.asarray(want).reshape(2, -1)):
            assert np.all(g == g[0])
            assert relmax(g, w) <= 1e-12
    if expansion:
        assert abs(sc.ap_half - ref.scale.ap) <= 1e-12 * ref.scale.ap


@pytest.mark.parametrize("kernel", ["auto", "generic"])
@pytest.mark.parametrize("dims,N", [(1, 100), (2, 40), (3, 20)])
def test_fp64_infinite_and_nan_sites_spread_as_in_the_oracle(gpu_capi, orc, dims, N, kernel):
    """Without expansion no sum sees them: after two steps the sites they have not
    reached are as they should be, and the others are not finite on either side."""
    q = (1.2,)
    f0, u0 = lattice_ics(dims, N, 20.0, 2, q=q, seed=3, amp=1e-2)
    f0, u0 = f0.reshape(2, -1).copy(), u0.reshape(2, -1)
    f0[0, 3], f0[1, N ** dims // 2] = np.inf, np.nan
    dt = courant_dt(dims, N, 20.0, 1.0, q)
    ref = orc.init(orc.Params(dims=dims, N=N, L=20.0, dt=dt, nf=2, q=q, expansion=False), np.ones_like(f0), u0)
    ref.f[...], ref.v[...] = f0.reshape(ref.f.shape), u0.reshape(ref.v.shape)
    orc.step(ref, 2)
    sc = gpu_capi.ce_scalars_t()
    sc.a = 1.0
    with gpu_capi.Simulation(dims=dims, N=N, L=20.0, dt=dt, nfields=2, q=q, expansion=False, kernel=kernel) as sim:
        sim.set_fields(f0, u0, gpu_capi.CE_VEL_STAGGERED, sc)
        sim.step(2)
        f, v, _ = sim.get_fields(gpu_capi.CE_VEL_STAGGERED)
    for got, want in ((f, ref.f), (v, ref.v)):
        got, want = got.reshape(-1), np.asarray(want).reshape(-1)
        finite = np.isfinite(want)
        assert 0 < (~finite).sum() < finite.size
        assert np.array_equal(np.isfinite(got), finite)
        assert relmax(got[finite], want[finite]) <= TOL64

