"""lbmd_set_types with fewer types than before, after the particles: a particle of a type that the new
table leaves out keeps that type's parameters, its fluid-side solvation force in the coupling velocity
included.  The same parameters in force, so the same bits as with the whole table."""
import numpy as np
import pytest

from gpu_common import Case, make_gpu, noisy_fluid

pytestmark = pytest.mark.gpu

TYPES = [(-0.2, 0.1, 0.0, 0.0, 1.0, 20.0), (-0.1, 0.05, 0.04, -0.03, 1.0, 20.0)]


def _case(substeps=1):
    dims = (18, 14, 16)
    rA, rB = noisy_fluid(dims, amp=0.03, seed=3)
    rng = np.random.default_rng(3)
    n = 60
    x = rng.uniform(0, 1, (n, 3)) * dims
    return Case(dims=dims, tau_r=0.9, g=1.2, seed=3, rhoA=rA, rhoB=rB, types=TYPES, x=x,
                v=rng.uniform(-0.02, 0.02, (n, 3)), ptype=(np.arange(n) % 2).astype(np.int32), q=np.zeros(n),
                md_substeps=substeps)


@pytest.mark.parametrize("substeps,passes", [(1, 2), (1, 1), (3, 2)])
def test_particles_keep_the_parameters_of_a_type_no_longer_listed(substeps, passes):
    from paper_1306_0788_gb300 import lbmd as L
    c = _case(substeps)
    got = []
    for listed in (1, 2):
        ctx = make_gpu(c, passes=passes)
        try:
            L.lbmd_set_types(ctx, [L.lbmd_ptype(*t) for t in TYPES[:listed]])
            L.lbmd_step(ctx, 4)
            f = np.stack([L.lbmd_get_populations(ctx, k, c.shape) for k in (0, 1)])
            got.append((f,) + L.lbmd_get_particles(ctx, c.n))
        finally:
            L.lbmd_destroy(ctx)
    for a, b in zip(*got):
        assert np.array_equal(a, b)


def test_batched_particles_keep_them_too():
    from paper_1306_0788_gb300 import lbmd as L
    from test_gpu_batch import add_case, read
    c = _case()
    b = L.lbmd_batch_create(0, L.LBMD_STORAGE_FP32, 4)
    try:
        slots = [add_case(b, c, 4) for _ in range(2)]
        L.lbmd_batch_set_types(b, slots[0], [L.lbmd_ptype(*TYPES[0])])
        L.lbmd_batch_step(b, 4)
        for x, y in zip(read(b, slots[0], c), read(b, slots[1], c)):
            assert np.array_equal(x, y)
    finally:
        L.lbmd_batch_destroy(b)
