"""Several handles of one kind whose lattices fit the resident kernel: each keeps its
own launch parameters, whatever is created or freed beside it, and tells whether it takes
that kernel."""
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


# (dims, N, fields, precision, expansion, takes the resident kernel), on both sides of
# each limit
ROUTES = [(3, 76, 2, "f64", True, True), (3, 77, 2, "f64", True, False), (2, 774, 1, "f64", False, True),
          (2, 775, 1, "f64", False, False), (1, 600000, 2, "f64", True, True), (1, 600001, 2, "f64", True, False),
          (3, 64, 2, "f32", True, True), (3, 65, 2, "f32", True, False), (3, 50, 4, "f32", True, True),
          (3, 51, 4, "f32", True, False), (2, 1048, 2, "f32", True, True), (2, 1049, 2, "f32", True, False),
          (1, 150000, 2, "f32", True, True), (1, 150001, 2, "f32", True, False), (3, 16, 1, "f32", True, False),
          (3, 32, 2, "f32", False, True), (3, 33, 2, "f32", False, False), (2, 599, 2, "f32", False, False),
          (2, 600, 2, "f32", False, True), (2, 836, 4, "f32", False, True), (2, 837, 4, "f32", False, False),
          (1, 1000, 2, "f32", False, False)]


@pytest.mark.parametrize("dims,N,nf,precision,expansion,resident", ROUTES)
def test_route_of_a_lattice_is_told(gpu_capi, dims, N, nf, precision, expansion, resident):
    with make(gpu_capi, dims, N, nf, precision, expansion) as sim:
        assert sim.resident == resident
        sim.step(2)
        sim.synchronize()
        assert sim.resident == resident
    with make(gpu_capi, dims, N, nf, precision, expansion, kernel="generic") as sim:
        assert not sim.resident
