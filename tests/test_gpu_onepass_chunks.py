"""The choice between one and two lattice passes, and the z-chunks of the one-pass update: chunk
counts that do not divide the depth, against the two-pass update (populations agree to a few FP32
roundings a step: 1e-6 of the largest after 6 steps)."""
import numpy as np
import pytest

from gpu_common import Case, make_gpu, noisy_fluid, pop_error, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,passes", [((80, 80, 80), 2), ((96, 96, 96), 1), ((100, 100, 100), 2),
                                         ((128, 128, 128), 1), ((256, 64, 128), 1)])
def test_passes_by_size(dims, passes):
    from paper_1306_0788_gb300 import lbmd as L
    ctx, _ = L.lbmd_create(L.params(dims, g_AB=1.2))
    try:
        assert L.lbmd_get_lattice_passes(ctx) == passes
    finally:
        L.lbmd_destroy(ctx)


@pytest.mark.parametrize("dims", [(40, 24, 37), (33, 9, 57), (64, 16, 8), (96, 96, 100), (128, 128, 59)])
def test_chunks_against_two_passes(dims):
    rA, rB = noisy_fluid(dims, amp=0.03, seed=3)
    u = np.random.default_rng(3).uniform(-0.02, 0.02, size=dims[::-1] + (3,))
    c = Case(dims=dims, tau_r=0.9, g=1.3, rhoA=rA, rhoB=rB, u=u)
    one, two = run_gpu(c, 6, passes=1)[0], run_gpu(c, 6, passes=2)[0]
    assert pop_error(one, two.astype(np.float64)) <= 1e-6
