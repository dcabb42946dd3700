"""The one-pass update with the fluctuating MRT collision, taken by size in FP32: against the two-pass
update, and its replayed graphs (whose noise counter is written into the update's nodes) against launches
one by one.  The two forms differ in the order of the density sums, a few FP32 roundings (6e-8 each, about
five in a population) a step: 2e-6 of the largest population after 6 steps."""
import numpy as np
import pytest

from gpu_common import Case, make_gpu, noisy_fluid, pop_error

pytestmark = pytest.mark.gpu


def _case(dims, n):
    rA, rB = noisy_fluid(dims, amp=0.03, seed=5)
    rng = np.random.default_rng(5)
    grid = np.stack(np.meshgrid(*[np.arange(4, d - 4, 8) for d in dims], indexing="ij"), -1).reshape(-1, 3)
    x = rng.permutation(grid)[:n] + rng.uniform(-1, 1, (n, 3))
    return Case(dims=dims, tau_r=0.9, g=1.3, kT=1e-5, seed=11, rhoA=rA, rhoB=rB, u=np.zeros(dims[::-1] + (3,)),
                collision=1, types=[(-1e-3, -2e-3, 0.0, 0.0, 1.0, 200.0)], wca={(0, 0): (1e-3, 1.0)}, x=x,
                v=np.zeros_like(x), ptype=np.zeros(n, dtype=np.int32), q=np.zeros(n))


def _run(c, steps, passes, graphs=True):
    from paper_1306_0788_gb300 import lbmd as L
    ctx = make_gpu(c, passes=passes)
    try:
        assert L.lbmd_get_lattice_passes(ctx) == (passes or 1)
        L.lbmd_set_graphs(ctx, graphs)
        L.lbmd_step(ctx, steps)
        f = np.stack([L.lbmd_get_populations(ctx, k, c.shape) for k in (0, 1)])
        return f, L.lbmd_get_particles(ctx, c.n)[0]
    finally:
        L.lbmd_destroy(ctx)


@pytest.mark.parametrize("dims,n", [((160, 152, 168), 500), ((191, 167, 170), 0)])
def test_onepass_mrt(dims, n):
    c = _case(dims, n)
    f1, x1 = _run(c, 6, 0)
    f2, x2 = _run(c, 6, 2)
    assert pop_error(f1, f2.astype(np.float64)) <= 2e-6
    assert n == 0 or np.abs(x1 - x2).max() <= 1e-6
    fd, xd = _run(c, 6, 0, graphs=False)
    assert np.array_equal(f1, fd) and np.array_equal(x1, xd)


def test_onepass_mrt_by_size_only():
    from paper_1306_0788_gb300 import lbmd as L
    ctx, _ = L.lbmd_create(L.params((32, 32, 32), g_AB=1.2, kT=1e-4, collision=L.LBMD_COLLISION_MRT))
    try:
        assert L.lbmd_get_lattice_passes(ctx) == 2
        with pytest.raises(L.LbmdError):
            L.lbmd_set_lattice_passes(ctx, 1)
    finally:
        L.lbmd_destroy(ctx)
