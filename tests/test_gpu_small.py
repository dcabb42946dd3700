"""Small lattices without particles: density pass and update in one launch give the bits of the two
passes -- tiles that do not divide the lattice, lattices thinner than a tile, the largest that takes
this form, every storage and collision."""
import numpy as np
import pytest

from gpu_common import Case, make_gpu, noisy_fluid

pytestmark = pytest.mark.gpu


def _state(c, passes, schedule):
    from paper_1306_0788_gb300 import lbmd as L
    ctx = make_gpu(c, passes=passes)
    try:
        for n in schedule:
            L.lbmd_step(ctx, n)
        return [L.lbmd_get_populations(ctx, k, c.shape) for k in range(2)] + list(L.lbmd_get_fields(ctx, c.shape))
    finally:
        L.lbmd_destroy(ctx)


@pytest.mark.parametrize("dims", [(1, 1, 1), (1, 2, 3), (16, 4, 4), (17, 5, 9), (2, 3, 40), (33, 30, 7), (64, 32, 32)])
@pytest.mark.parametrize("storage,collision", [(0, 0), (0, 1), (1, 0), (2, 1)])
def test_one_launch_gives_the_bits_of_two_passes(dims, storage, collision):
    rA, rB = noisy_fluid(dims, amp=0.02, seed=3)
    u = np.random.default_rng(3).uniform(-0.02, 0.02, size=dims[::-1] + (3,))
    c = Case(dims=dims, tau_r=0.9, g=1.2, kT=1e-4, seed=5, rhoA=rA, rhoB=rB, u=u, storage=storage,
             collision=collision, rho0=(1.0, 1.0))
    for a, b in zip(_state(c, 0, (3, 2)), _state(c, 2, (3, 2))):
        assert np.array_equal(a, b)
