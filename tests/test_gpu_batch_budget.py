"""What a replica with particles is charged against the batch's memory budget covers what the batch allocates
for them: particle arrays with a quarter of slack, rows, and in FP32 the two sets of node bits with a
quarter of slack, a whole word per row at least (the larger part of it on a lattice of few columns)."""
import re

import pytest

pytestmark = pytest.mark.gpu


def _needed(L, dims, storage, np_max):
    b = L.lbmd_batch_create(1, storage, 2)  # a budget of one byte: refused, with the bytes it would take
    try:
        with pytest.raises(L.LbmdError) as e:
            L.lbmd_batch_add(b, L.params(dims, storage=storage, rho0=(1.0, 1.0)), np_max, 1)
        assert e.value.code == L.LBMD_E_NOMEM
        return int(re.search(r"needs (\d+) bytes", str(e.value)).group(1))
    finally:
        L.lbmd_batch_destroy(b)


@pytest.mark.parametrize("dims", [(4, 64, 48), (33, 20, 17), (128, 128, 128)])
@pytest.mark.parametrize("storage", [0, 1])
def test_particle_share_covers_the_node_bits(dims, storage):
    from paper_1306_0788_gb300 import lbmd as L
    particles = 40
    nx, ny, nz = dims
    share = _needed(L, dims, storage, particles) - _needed(L, dims, storage, 0)
    arrays = 2 * (16 + 16 + 16 + 4) + 6 * 16 + 3 * 4  # two sets of particles, six forces, three index arrays
    bits = 2 * ny * nz * ((nx + 31) // 32) * 4 if storage == L.LBMD_STORAGE_FP32 else 0
    assert share >= 1.25 * particles * arrays + 3 * 4 * ny * nz + 1.25 * bits
