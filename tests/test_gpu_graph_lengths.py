"""The longer step graphs, recorded after 128 and 4096 replayed steps: calls of every size around
their lengths give the bits of launches one by one.  (A flat interface at coexistence with heavy
particles, the model of the served replicas: stable for thousands of steps.)"""
import numpy as np
import pytest

from gpu_common import Case, make_gpu
from paper_1306_0788_gb300 import inputs

pytestmark = pytest.mark.gpu


def _case(particles, dims=(16, 14, 18), **more):
    rA, rB = inputs.flat_slab(dims, 1.8586, 0.1414)  # coexistence at g rho = 1.5
    x = inputs.spaced_particles(particles, dims, 2.5, seed=4)
    c = Case(dims=dims, g=1.5, kT=1e-4, seed=9, rhoA=rA, rhoB=rB, x=x, v=np.zeros_like(x),
             ptype=np.zeros(particles, dtype=np.int32), types=[(0.0, 0.0, 0.0, 0.0, 1.0, 200.0)],
             wca={(0, 0): (1.0, 1.0)})
    for k, v in more.items():
        setattr(c, k, v)
    return c


def _run(c, graphs, schedule):
    from paper_1306_0788_gb300 import lbmd as L
    ctx = make_gpu(c)
    try:
        L.lbmd_set_graphs(ctx, graphs)
        for n in schedule:
            L.lbmd_step(ctx, n)
        f = np.stack([L.lbmd_get_populations(ctx, k, c.shape) for k in range(2)])
        return (f, L.lbmd_step_count(ctx)) + L.lbmd_get_particles(ctx, c.n)
    finally:
        L.lbmd_destroy(ctx)


@pytest.mark.parametrize("c,schedule", [(_case(40), (130, 7, 8, 9, 21)),
                                        (_case(40, collision=1), (129, 10, 3, 40)),
                                        (_case(40, md_substeps=3), (128, 11, 16)),
                                        (_case(40, storage=1, rho0=(1.0, 1.0)), (130, 17)),
                                        (_case(0), (4100, 31, 32, 33, 75))])
def test_long_graphs_are_bit_identical(c, schedule):
    a, b = _run(c, True, schedule), _run(c, False, schedule)
    assert a[1] == b[1] == sum(schedule)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("nz,storage,collision", [(64, 0, 1), (63, 0, 1), (64, 1, 0)])
def test_large_and_small_update_blocks(nz, storage, collision):
    """From 2^19 nodes (128 x 64 x 64) the update runs in blocks of 64 threads: its noise counter is
    patched in the graphs as that of the 256-thread one below."""
    c = _case(300, dims=(128, 64, nz), storage=storage, collision=collision, rho0=(1.0, 1.0))
    a, b = _run(c, True, (3, 4)), _run(c, False, (3, 4))
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
