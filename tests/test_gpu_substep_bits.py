"""MD sub-stepping's node marks are cleared by the cells that were marked, not by a sweep over the lattice by
however many blocks the particles give: a step with few particles takes no longer than one with many.  And
none is left behind or missing as particles move: the same bits as in a context without a past."""
import time

import numpy as np
import pytest

from gpu_common import Case, make_gpu, noisy_fluid

pytestmark = pytest.mark.gpu


def _case(dims, n, substeps, speed=0.0):
    rng = np.random.default_rng(n)
    rA, rB = noisy_fluid(dims, amp=0.01, seed=2)
    return Case(dims=dims, g=0.5, rhoA=rA, rhoB=rB, types=[(0.0, 0.0, 0.0, 0.0, 0.01, 200.0)],
                x=rng.uniform(0, 1, (n, 3)) * dims, v=rng.uniform(-speed, speed, (n, 3)),
                ptype=np.zeros(n, dtype=np.int32), q=np.zeros(n), md_substeps=substeps)


def _step_time(n):
    from paper_1306_0788_gb300 import lbmd as L
    ctx = make_gpu(_case((2, 1024, 2048), n, 4))  # a word per row of two columns: 2 M words
    try:
        times = []
        for _ in range(6):
            t = time.perf_counter()
            L.lbmd_step(ctx, 20)
            L.lbmd_sync(ctx)
            times.append(time.perf_counter() - t)
        return min(times[1:])
    finally:
        L.lbmd_destroy(ctx)


def test_few_particles_take_no_longer_than_many():
    few, many = _step_time(8), _step_time(800)
    print("us a step: %.0f with 8 particles, %.0f with 800" % (few * 5e4, many * 5e4))
    assert few <= 1.05 * many


@pytest.mark.parametrize("n", [1, 9, 200])
def test_marks_follow_the_particles(n):
    """Ten steps in one context against a fresh context for each, with particles that cross a cell in a step
    or two and numbers of particles that change in between."""
    from paper_1306_0788_gb300 import lbmd as L
    c = _case((9, 37, 33), n, 3, speed=0.8)
    more = _case((9, 37, 33), 3 * n + 5, 3, speed=0.8)

    def state(ctx, k):
        return [L.lbmd_get_populations(ctx, z, c.shape) for z in (0, 1)] + list(L.lbmd_get_particles(ctx, k))

    ctx = make_gpu(c)
    try:
        for turn, p in enumerate((c, more, c)):
            if turn:
                L.lbmd_set_particles(ctx, p.x, p.v, p.ptype, p.q)
            for _ in range(4):
                before = state(ctx, p.n)
                L.lbmd_step(ctx, 1)
                after = state(ctx, p.n)
                fresh = make_gpu(p)
                try:
                    for z in (0, 1):
                        L.lbmd_set_populations(fresh, z, before[z])
                    L.lbmd_set_particles(fresh, before[2], before[3], p.ptype, p.q)
                    L.lbmd_step(fresh, 1)
                    for a, b in zip(after, state(fresh, p.n)):
                        assert np.array_equal(a, b)
                finally:
                    L.lbmd_destroy(fresh)
    finally:
        L.lbmd_destroy(ctx)
