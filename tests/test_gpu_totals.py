"""The FP64 totals against exactly rounded sums of the same populations (math.fsum): the device adds
groups of nodes without rounding error to about 48 bits and the groups in FP64, so a total is off by
at most the FP64 roundings on the way, about 50 at the sizes here: 5e-15 of the mass."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
              (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
              (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)])


@pytest.mark.parametrize("dims", [(1, 1, 1), (7, 5, 3), (40, 33, 29), (101, 96, 67)])
def test_totals_are_the_sums_of_the_populations(dims):
    from paper_1306_0788_gb300 import lbmd as L
    g = np.random.default_rng(sum(dims))
    shape = dims[::-1]
    rho = [(10.0 ** g.uniform(-2, 2, size=shape)).astype(np.float32) for _ in range(2)]
    u = g.uniform(-0.1, 0.1, size=shape + (3,)).astype(np.float32)
    ctx, _ = L.lbmd_create(L.params(dims, g_AB=1.0))
    try:
        L.lbmd_init_fluid(ctx, *rho, u)
        d = L.lbmd_diagnostics(ctx)
        f = [L.lbmd_get_populations(ctx, k, shape).astype(np.float64).reshape(19, -1) for k in range(2)]
    finally:
        L.lbmd_destroy(ctx)
    mass = [math.fsum(x.ravel()) for x in f]
    momentum = [math.fsum(((f[0] + f[1]) * C[:, a:a + 1]).ravel()) for a in range(3)]
    assert np.abs(d[:2] - mass).max() <= 5e-15 * max(mass)
    assert np.abs(d[2:5] - momentum).max() <= 5e-15 * sum(mass)
