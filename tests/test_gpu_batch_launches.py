"""A batch step launches the particle kernels only while some replica has particles: five kernels a step
without (density pass, update, step count, two of the drift check), fifteen with.  Replicas come out the
same either way, also where the batch changes between the two."""
import numpy as np
import pytest

from test_gpu_batch import add_case, coupled_case, fluid_case, read, run_alone, same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [0, 1])
def test_no_particle_kernels_without_particles(storage):
    from paper_1306_0788_gb300 import lbmd as L
    rho0 = (1.0, 1.0) if storage else (0.0, 0.0)
    fluid, coupled = fluid_case((20, 14, 18), 3), coupled_case((16, 12, 14), 40, seed=4)
    b = L.lbmd_batch_create(0, storage, 4)

    def step(n):
        before = L.lbmd_batch_launch_count(b)
        L.lbmd_batch_step(b, n)
        return (L.lbmd_batch_launch_count(b) - before) / n

    try:
        s = add_case(b, fluid, 12, storage=storage, rho0=rho0)
        assert step(4) == 5
        t = add_case(b, coupled, 4, storage=storage, rho0=rho0)
        L.lbmd_batch_poll(b, 4)
        assert 15 <= step(4) <= 16  # and the launches of the new layout
        with_particles = read(b, t, coupled)
        L.lbmd_batch_remove(b, t)
        assert step(4) == 5
        assert same(read(b, s, fluid)[:1], run_alone(fluid, 12, storage=storage, rho0=rho0)[:1])
        assert same(with_particles, run_alone(coupled, 4, storage=storage, rho0=rho0))
    finally:
        L.lbmd_batch_destroy(b)
