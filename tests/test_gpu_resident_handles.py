"""Several handles of one kind whose lattices fit the resident kernel: each keeps its
own launch parameters, whatever is created or freed beside it."""
import numpy as np
import pytest

from test_gpu_resident import make, state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,dims,sizes", [("f32", 3, (64, 32, 16)), ("f64", 3, (64, 32, 16)),
                                                  ("f32", 2, (500, 64)), ("f64", 2, (500, 64)),
                                                  ("f32", 1, (120000, 1000)), ("f64", 1, (300000, 1000))])
def test_lattices_of_several_sizes_side_by_side(gpu_capi, precision, dims, sizes):
    """The largest is created first: what the smaller ones ask of the kernel must not
    take from it.  Each ends where it ends alone."""
    capi = gpu_capi
    alone = []
    for N in sizes:
        with make(capi, dims, N, 2, precision, True) as sim:
            sim.step(60)
            alone.append(state(capi, sim)[:2])
    sims = [make(capi, dims, N, 2, precision, True) for N in sizes]
    try:
        for _ in range(3):
            for s in sims:
                s.step(20)
        with make(capi, dims, 9, 2, precision, True) as another:
            another.step(5)
            for s, (f, v) in zip(sims, alone):
                fs, vs, sc = state(capi, s)
                assert sc.step == 60 and np.array_equal(fs, f) and np.array_equal(vs, v)
                s.step(1)
                s.synchronize()
    finally:
        for s in sims:
            s.close()

