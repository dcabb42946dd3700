"""The precision of the FP64 totals where large momenta cancel within the group of nodes that a thread adds up
before it goes over to FP64."""
import math

import numpy as np
import pytest

from test_gpu_totals import C

pytestmark = pytest.mark.gpu


def test_groups_of_nodes_keep_the_precision_of_fp64():
    """Momenta that cancel between the nodes that one thread sums: layers of heavy fluid moving one way and the
    other along x and y, light fluid between, of intermediate density next to them.  (A node of heavy
    populations, up to 2^17 in sum, and populations of densities from 100, at least 1 each, needs 17 + 24 of
    the 48 bits of the device's pairs: node totals are exact.)  Added in FP64, a light node's
    total rounds by at most half a unit in the last place of a heavy node's momentum, 12^-1/2 of a unit in
    the mean: six standard deviations of N / 2 of them.  (A pair carried over several nodes holds 48 bits and
    misses that by a factor of about twenty.)"""
    from paper_1306_0788_gb300 import lbmd as L
    dims = (76, 64, 80)
    shape = dims[::-1]
    g = np.random.default_rng(20)
    rho = [(10.0 ** g.uniform(-5, -3, size=shape)).astype(np.float32) for _ in range(2)]
    u = g.uniform(-0.1, 0.1, size=shape + (3,)).astype(np.float32)
    for r in rho:
        for layer, decade in ((20, 2), (21, 0), (38, 0), (39, 2)):
            r[layer::40] = 10.0 ** g.uniform(decade, decade + 1, size=r[layer::40].shape)
        r[0:20] = r[40:60] = 2.0 ** 20
    u[0:20] = (0.05, 0.03, 0.0)
    u[40:60] = (-0.05, -0.03, 0.0)
    ctx, _ = L.lbmd_create(L.params(dims, g_AB=1.0))
    try:
        L.lbmd_init_fluid(ctx, *rho, u)
        d = L.lbmd_diagnostics(ctx)
        f = [L.lbmd_get_populations(ctx, k, shape).astype(np.float64).reshape(19, -1) for k in range(2)]
    finally:
        L.lbmd_destroy(ctx)
    for a, ua in enumerate((0.05, 0.03)):
        momentum = math.fsum(((f[0] + f[1]) * C[:, a:a + 1]).ravel())
        unit = np.spacing(2 * 2.0 ** 20 * ua)
        assert abs(d[2 + a] - momentum) <= 6 * math.sqrt(0.5 * f[0].shape[1] / 12) * unit
