"""Bounded waits of the resident kernel and of the 3D FP64 kernel that run out: with
CE_FLAG_TEST_WAIT_STALL one launch waits for an arrival that never comes, gives up after
~0.5 ms, latches CE_ETIMEOUT and completes.  The context stays usable, and the handle
recovers with the next ce_set_fields (the flag holds for one launch)."""
import numpy as np
import pytest

from paper_0712_0813_gb300.icgen import courant_dt, lattice_ics

pytestmark = pytest.mark.gpu

Q = (1.2,)


def config(dims, N, precision, expansion):
    return dict(dims=dims, N=N, L=20.0, dt=0.9 * courant_dt(dims, N, 20.0, 1.0, Q), nfields=2, q=Q,
                expansion=expansion, precision=precision)


def run(capi, cfg, f0, u0, steps):
    with capi.Simulation(**cfg) as sim:
        sim.set_fields(f0, u0)
        sim.step(steps)
        return sim.get_fields(capi.CE_VEL_STAGGERED)


def expect(capi, code, call, *args):
    with pytest.raises(capi.CeError) as ei:
        call(*args)
    assert ei.value.code == code


@pytest.mark.parametrize("dims,N,precision,expansion", [(3, 24, "f32", True), (3, 24, "f32", False), (2, 60, "f64", True),
                                                        (1, 5000, "f64", False), (1, 5000, "f32", True)])
def test_resident_kernel_gives_up_and_recovers(gpu_capi, dims, N, precision, expansion):
    capi = gpu_capi
    f0, u0 = lattice_ics(dims, N, 20.0, 2, q=Q, seed=2)
    cfg = config(dims, N, precision, expansion)
    good = run(capi, cfg, f0, u0, 50)
    with capi.Simulation(**cfg, flags=capi.CE_FLAG_TEST_WAIT_STALL) as bad:
        assert bad.resident
        bad.set_fields(f0, u0)
        bad.step(10)
        expect(capi, capi.CE_ETIMEOUT, bad.synchronize)
        expect(capi, capi.CE_ETIMEOUT, bad.energy)   # the code stays latched
        bad.set_fields(f0, u0)
        bad.step(50)
        f, v, sc = bad.get_fields(capi.CE_VEL_STAGGERED)
    assert sc.step == 50 and sc.a == good[2].a
    assert np.array_equal(f, good[0]) and np.array_equal(v, good[1])


@pytest.mark.parametrize("expansion", [True, False])
@pytest.mark.parametrize("N,nf", [(24, 2), (37, 4)])
def test_fp64_kernel_gives_up_and_recovers(gpu_capi, N, nf, expansion):
    capi = gpu_capi
    q = (0.8, 5.0, 40.0)[:nf - 1]
    f0, u0 = lattice_ics(3, N, 20.0, nf, q=q, seed=2)
    cfg = dict(dims=3, N=N, L=20.0, dt=0.9 * courant_dt(3, N, 20.0, 1.0, q), nfields=nf, q=q, expansion=expansion,
               kernel="generic")
    good = run(capi, cfg, f0, u0, 5)
    with capi.Simulation(**cfg, flags=capi.CE_FLAG_TEST_WAIT_STALL) as bad:
        expect(capi, capi.CE_ETIMEOUT, bad.set_fields, f0, u0)   # the start-up half kick
        expect(capi, capi.CE_ESTATE, bad.step, 1)
        bad.set_fields(f0, u0)
        bad.step(5)
        f, v, _ = bad.get_fields(capi.CE_VEL_STAGGERED)
    assert np.array_equal(f, good[0]) and np.array_equal(v, good[1])
