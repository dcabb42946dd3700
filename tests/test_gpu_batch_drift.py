"""The drift figures of a replica (FP64 sums compared with its reference) are the same bits alone, in mixes
of other replicas that join and leave between the reference and the check, and with any tile size.  The
densities span four decades, so that the FP64 sums round (those of a nearly uniform fluid are exact in any
grouping)."""
import numpy as np
import pytest

from test_gpu_batch import fluid_case

pytestmark = pytest.mark.gpu

DIMS = (64, 33, 29)


def _decades():
    """1e-4 to 1 along x, the same in both components, times 1 +- 0.03 at random."""
    c = fluid_case(DIMS, 9, g=0.0)
    c.rhoA, c.rhoB = (r * 10.0 ** (2 * np.cos(2 * np.pi * np.arange(DIMS[0]) / DIMS[0]) - 2) for r in (c.rhoA, c.rhoB))
    return c


def _add(L, b, c, storage, total, every):
    s, _ = L.lbmd_batch_add(b, L.params(c.dims, g_AB=c.g, storage=storage, rho0=(0.01, 0.01), diag_every=every,
                                        drift_tol=0.1 if every else 0.0), 0, total)
    a, bb, u = c.fields32()
    L.lbmd_batch_init_fluid(b, s, a, bb, u)
    return s


def _drift(storage, others=(), config=None, leave=False):
    """Drift after 8 steps in two calls of 4; `others`: edges of replicas that join between the two."""
    from paper_1306_0788_gb300 import lbmd as L
    b = L.lbmd_batch_create(0, storage, 64)
    try:
        if config:
            L.lbmd_batch_set_config(b, *config)
        s = _add(L, b, _decades(), storage, 8, 4)
        L.lbmd_batch_step(b, 4)
        joined = [_add(L, b, fluid_case((e,) * 3, e), storage, 4, 0) for e in others]
        L.lbmd_batch_step(b, 3)
        if leave:
            for t in joined:
                L.lbmd_batch_remove(b, t)
        L.lbmd_batch_step(b, 1)
        L.lbmd_batch_poll(b, 64)
        d = L.lbmd_batch_get_drift(b, s)
        assert d[0] == 8 and d[4] == 2
        return d
    finally:
        L.lbmd_batch_destroy(b)


@pytest.mark.parametrize("storage", [0, 1])
def test_drift_does_not_depend_on_the_mix_or_the_tiles(storage):
    alone = _drift(storage)
    assert max(alone[1:4]) > 0
    for other in (_drift(storage, others=(100, 90, 16)), _drift(storage, others=(100,), leave=True),
                  _drift(storage, config=(256, 100, 100, 3)), _drift(storage, config=(4096, 50, 60, 2))):
        assert np.array_equal(alone, other)
