"""The resident multi-step kernel (small lattices on the automatic choice) against
the kernels that take one launch a step, at the sizes where its bricks, halos and
chunks can go wrong, and its behaviour under repeated, chunked, concurrent and
captured calls."""
import threading

import numpy as np
import pytest

from paper_0712_0813_gb300.icgen import courant_dt

pytestmark = pytest.mark.gpu

L = 20.0
Q = (0.8, 5.0, 40.0)


def make(capi, dims, N, nf, precision, expansion, kernel="auto", seed=3, **kw):
    rng = np.random.default_rng([seed, dims, N, nf])
    f0 = 1e-2 * rng.standard_normal((nf, N ** dims))
    f0[0] += 1.0
    u0 = 1e-2 * rng.standard_normal((nf, N ** dims))
    q = Q[:nf - 1]
    sim = capi.Simulation(dims=dims, N=N, L=L, dt=courant_dt(dims, N, L, 1.0, q), nfields=nf, q=q,
                          expansion=expansion, precision=precision, kernel=kernel, **kw)
    sim.set_fields(f0, u0)
    return sim


def state(capi, sim):
    return sim.get_fields(capi.CE_VEL_STAGGERED)


# one-site bricks, uneven last bricks, bricks as wide as the lattice, a block with
# many sites a thread, the largest lattices that take the kernel
SHAPES = [(1, 3), (1, 153), (1, 4099), (1, 262144), (2, 3), (2, 31), (2, 257), (2, 700), (3, 3), (3, 5), (3, 33),
          (3, 64), (3, 80)]


@pytest.mark.parametrize("nf", [1, 2, 3, 4])
@pytest.mark.parametrize("dims,N", SHAPES)
def test_fp32_fields_equal_the_generic_kernel(gpu_capi, dims, N, nf):
    """Without expansion every FP32 kernel does the same operations at a site."""
    with make(gpu_capi, dims, N, nf, "f32", False) as a, make(gpu_capi, dims, N, nf, "f32", False, "generic") as b:
        for n in (1, 2, 9):
            a.step(n)
            b.step(n)
        fa, va, sa = state(gpu_capi, a)
        fb, vb, sb = state(gpu_capi, b)
        assert np.array_equal(fa, fb) and np.array_equal(va, vb)
        assert sa.step == sb.step == 12 and sa.t == sb.t


@pytest.mark.parametrize("precision,eps,sums", [("f32", 2.0 ** -24, 1e-6), ("f64", 2.0 ** -53, 1e-13)])
@pytest.mark.parametrize("dims,N,nf", [(1, 4099, 2), (2, 257, 2), (3, 5, 3), (3, 33, 2), (3, 64, 4)])
def test_one_expanding_step_against_the_generic_kernel(gpu_capi, dims, N, nf, precision, eps, sums):
    """One step from the same state: f' is the same but for FP64's grouping (none: both
    form it by the same two FMAs); a'' carries the sums' order (FP32 partials: 1e-6 of
    the source, FP64: rounding), v' = w + c f that order times c f and rounding."""
    with make(gpu_capi, dims, N, nf, precision, True) as a, make(gpu_capi, dims, N, nf, precision, True, "generic") as b:
        a.step(1)
        b.step(1)
        fa, va, sa = state(gpu_capi, a)
        fb, vb, sb = state(gpu_capi, b)
        assert np.array_equal(fa, fb)
        assert abs(sa.app - sb.app) <= sums * (abs(sb.app) + sb.ap_half ** 2)
        assert sa.a == pytest.approx(sb.a, rel=4 * 2.0 ** -53)
        dx2 = (N / L) ** 2
        dt = courant_dt(dims, N, L, 1.0, Q[:nf - 1])
        scale = np.abs(vb).max() + dt * (4 * dims * dx2 + 1) * np.abs(fb).max()
        assert np.abs(va - vb).max() <= (sums + 8 * eps) * scale


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("dims,N,expansion", [(3, 17, True), (2, 40, False), (1, 1000, True)])
def test_chunks_of_steps_give_the_same_bits(gpu_capi, dims, N, expansion, precision):
    """One call, many calls, and a call longer than one launch (4096 steps)."""
    with make(gpu_capi, dims, N, 2, precision, expansion) as a, make(gpu_capi, dims, N, 2, precision, expansion) as b:
        a.step(4200)
        for n in (1, 31, 32, 33, 4000, 103):
            b.step(n)
        fa, va, sa = state(gpu_capi, a)
        fb, vb, sb = state(gpu_capi, b)
        assert np.array_equal(fa, fb) and np.array_equal(va, vb)
        assert (sa.a, sa.ap_half, sa.app, sa.step) == (sb.a, sb.ap_half, sb.app, sb.step)


def test_concurrent_handles(gpu_capi):
    """Handles stepped from several threads, each on its own stream, end where they
    end alone."""
    capi = gpu_capi
    specs = [(3, 32, "f64"), (3, 48, "f32"), (2, 300, "f32"), (1, 5000, "f64")]
    alone = []
    for dims, N, precision in specs:
        with make(capi, dims, N, 2, precision, True) as sim:
            sim.step(3000)
            alone.append(state(capi, sim)[:2])
    sims = [make(capi, dims, N, 2, precision, True) for dims, N, precision in specs]
    try:
        def work(sim):
            for _ in range(30):
                sim.step(100)
        threads = [threading.Thread(target=work, args=(s,)) for s in sims]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for sim, (f, v) in zip(sims, alone):
            fs, vs, sc = state(capi, sim)
            assert sc.step == 3000 and np.array_equal(fs, f) and np.array_equal(vs, v)
    finally:
        for s in sims:
            s.close()


def test_steps_captured_by_the_caller_replay(gpu_capi):
    """Steps recorded into the caller's own graph take plain launches, so every
    replay advances the lattice by them."""
    import torch
    capi = gpu_capi
    st = torch.cuda.Stream()
    with make(capi, 3, 24, 2, "f32", True, stream=st.cuda_stream) as a, make(capi, 3, 24, 2, "f32", True) as b:
        a.step(4)
        a.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            a.step(2)
        with torch.cuda.stream(st):
            for _ in range(5):
                g.replay()
        st.synchronize()
        b.step(14)
        fa, va, _ = state(capi, a)
        fb, vb, _ = state(capi, b)
        # other kernels, so another order of the sums: FP32 rounding over ten steps
        assert np.abs(fa - fb).max() <= 1e-5 * np.abs(fb).max()
        assert np.abs(va - vb).max() <= 1e-4 * np.abs(vb).max()
