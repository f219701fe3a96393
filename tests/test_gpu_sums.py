"""The read-outs' sums at the sizes where their kernels change shape: the diagnostics
pass (energies, means, variances) over sides that leave ragged segments and chunks,
and the allocation-free moments across their two forms (FP64 sums below 2^17 sites of
an FP32 array, float pairs from there) and outside the pairs' range."""
import numpy as np
import pytest

from paper_0712_0813_gb300.icgen import courant_dt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("nf", [1, 2, 4])
@pytest.mark.parametrize("dims,N", [(1, 3), (1, 4095), (1, 4097), (2, 3), (2, 31), (2, 257), (3, 3), (3, 8), (3, 33),
                                    (3, 66)])
def test_diagnostics_against_numpy(gpu_capi, dims, N, nf, precision):
    """K, G, V, E, means and variances of the downloaded state, formed in FP64.

    Tolerances: per-site terms are rounded in the storage type (unit u), a thread adds
    16 of them in it, so each positive sum is within ~20 u of itself; in FP32 a term's
    own inputs carry rounding too: u_i (the synchronised velocity) of u times the
    Laplacian's weights, included as u_scale."""
    capi = gpu_capi
    L, q = 20.0, (0.8, 5.0, 40.0)[:nf - 1]
    dt = courant_dt(dims, N, L, 1.0, q)
    rng = np.random.default_rng([dims, N, nf])
    f0 = 0.1 * rng.standard_normal((nf, N ** dims))
    f0[0] += 1.0
    u0 = 0.1 * rng.standard_normal((nf, N ** dims))
    with capi.Simulation(dims=dims, N=N, L=L, dt=dt, nfields=nf, q=q, expansion=True, precision=precision) as sim:
        sim.set_fields(f0, u0)
        sim.step(3)
        e = sim.energy()
        mean, var = sim.means_variances()
        f, us, _ = sim.get_fields(capi.CE_VEL_SYNC)
    f, us = f.reshape((nf,) + (N,) * dims), us.reshape(nf, -1)
    eps = 2.0 ** -24 if precision == "f32" else 2.0 ** -53
    dx2 = (N / L) ** 2
    G = [0.5 * dx2 * sum(((np.roll(x, -1, d) - x) ** 2).mean() for d in range(dims)) for x in f]
    K = 0.5 * (us ** 2).mean(1)
    V = (f[0] ** 2 * (0.25 * f[0] ** 2 + 0.5 * sum(qi * x ** 2 for qi, x in zip(q, f[1:])))).mean()
    u_scale = eps * dt * (4 * dims + 2) * dx2 * np.abs(f).max() / max(np.abs(us).max(), 1e-30)
    tol = 20 * eps + 4 * u_scale
    np.testing.assert_allclose(e["K"], K, rtol=tol)
    np.testing.assert_allclose(e["G"], G, rtol=20 * eps + 4 * eps * np.abs(f).max() / 0.1)
    assert e["V"] == pytest.approx(V, rel=20 * eps)
    assert e["E"] == pytest.approx(K.sum() + sum(G) + V, rel=2 * tol)
    x = f.reshape(nf, -1)
    spread = np.abs(x - x[:, :1]).max(1)
    assert np.all(np.abs(mean - x.mean(1)) <= 20 * eps * spread + 4 * 2.0 ** -53 * np.abs(x).max(1))
    assert np.all(np.abs(var - x.var(1)) <= 40 * eps * spread ** 2)


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("n", [1, 7, 2047, 2049, (1 << 17) - 1, 1 << 17, (1 << 17) + 5, 400001])
def test_moments_sizes(gpu_capi, n, precision):
    """Fields of ordinary, tiny and huge spread; an infinity and a NaN."""
    import torch
    capi = gpu_capi
    rng = np.random.default_rng(n)
    dtype = np.float32 if precision == "f32" else np.float64
    x = rng.standard_normal((4, n))
    x = np.stack([1.0 + 1e-3 * x[0], 1e-3 * x[1], 1e-16 * x[2], 1e17 * x[3]]).astype(dtype)

    def moments(a):
        d = torch.tensor(a, device="cuda")
        mean = torch.empty(4, dtype=torch.float64, device="cuda")
        var = torch.empty(4, dtype=torch.float64, device="cuda")
        capi.ce_moments_noalloc(d.data_ptr(), capi.CE_F32 if precision == "f32" else capi.CE_F64, n, 4,
                                torch.cuda.current_stream().cuda_stream, mean.data_ptr(), var.data_ptr())
        torch.cuda.synchronize()
        return mean.cpu().numpy(), var.cpu().numpy()

    mean, var = moments(x)
    y = x.astype(np.longdouble)
    spread = np.abs(y - y[:, :1]).max(1)
    # FP64 sums, or sums as accurate: rounding of n terms, and of the final operations
    tol = 2.0 ** -50
    assert np.all(np.abs(mean - y.mean(1)) <= tol * (spread + np.abs(y[:, 0])))
    assert np.all(np.abs(var - y.var(1)) <= 4 * tol * spread ** 2)
    if n > 7:
        x[0, n // 2], x[1, n - 1] = np.inf, np.nan
        mean, var = moments(x)
        assert np.isinf(mean[0]) and np.isnan(var[0]) and np.isnan(mean[1]) and np.isnan(var[1])
        assert np.isfinite(mean[2:]).all() and np.isfinite(var[2:]).all()
