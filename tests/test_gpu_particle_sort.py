"""The particle sort at the edges of its two forms -- one block (up to 8192 rows and 4096 particles)
and the chain of launches beyond -- with crowded rows and particles that change rows, against the
FP64 oracle (tolerances of the parity tests: populations 1e-5, positions 1e-4)."""
import numpy as np
import pytest

from gpu_common import Case, noisy_fluid, pop_error, position_error, run_gpu, run_oracle
from paper_1306_0788_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,n", [((5, 64, 128), 300),     # 8192 rows: one block
                                    ((6, 91, 91), 300),      # 8281 rows: the chain
                                    ((64, 16, 16), 4096),    # 16 particles a row: one block
                                    ((64, 16, 16), 4097)])   # the chain
def test_sort_forms_against_the_oracle(dims, n):
    rA, rB = noisy_fluid(dims, seed=n)
    x = inputs.spaced_particles(n, dims, 1.25, seed=n + 1)
    v = np.random.default_rng(n).uniform(-0.4, 0.4, size=(n, 3))
    c = Case(dims=dims, g=1.2, kT=1e-4, rhoA=rA, rhoB=rB, x=x, v=v, ptype=np.zeros(n, dtype=np.int32),
             types=[(-0.01, 0.01, 0.002, 0.0, 0.2, 50.0)])
    fg, xg, vg, _ = run_gpu(c, 4)
    fo, xo, vo, _ = run_oracle(c, 4)
    assert pop_error(fg, fo) <= 1e-5
    assert position_error(xg, xo, c.x, c.dims) <= 1e-4
    assert np.abs(vg - vo).max() <= 1e-4 * np.abs(vo).max()


@pytest.mark.parametrize("nz", [128, 127])
def test_coupling_reads_marked_nodes(nz):
    """From 2^22 nodes (256 x 128 x 128) two passes store j' only at the corners of the particles' cells;
    one pass forms it at the particles: the particles agree to a few FP32 roundings a step (velocities 1e-5
    of the largest after 4 steps), those in the periodic edge cells among them."""
    dims, n = (256, 128, nz), 3000
    rA, rB = noisy_fluid(dims, amp=0.02, seed=8)
    u = np.random.default_rng(8).uniform(-0.05, 0.05, size=dims[::-1] + (3,))
    x = np.random.default_rng(9).uniform(0, 1, size=(n, 3)) * dims
    x[:200, 0] = dims[0] - 0.5 * np.random.default_rng(10).random(200)
    x[200:400, 2] = dims[2] - 0.5 * np.random.default_rng(11).random(200)
    c = Case(dims=dims, g=1.2, rhoA=rA, rhoB=rB, u=u, x=x, v=np.random.default_rng(12).uniform(-0.4, 0.4, size=(n, 3)),
             ptype=np.zeros(n, dtype=np.int32), types=[(-0.01, 0.01, 0.002, 0.0, 0.2, 50.0)])
    _, _, v1, _ = run_gpu(c, 4, passes=1)
    _, _, v2, _ = run_gpu(c, 4, passes=2)
    assert np.abs(v1 - v2).max() <= 1e-5 * np.abs(v1).max()
