"""The longer step graphs with everything in them: 32 steps with particles on the side stream and noise
counters written into their nodes, 8 steps of the one-pass update, whose corner j' crosses from step to
step on the side stream.  The bits of launches one by one.  And the one-pass update with the fluctuating
MRT collision, taken by size, where its tiles have one column or one row (densities pulled instead of
summed): the two-pass update's populations up to the order of the density sums, as test_gpu_onepass_mrt."""
import numpy as np
import pytest

from gpu_common import pop_error
from test_gpu_graph_lengths import _case, _run
from test_gpu_onepass_mrt import _case as mrt_case
from test_gpu_onepass_mrt import _run as run_passes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("substeps,collision", [(1, 1), (1, 0), (3, 0)])
def test_graphs_of_32_steps_with_particles(substeps, collision):
    c = _case(40, collision=collision, md_substeps=substeps)
    schedule = (4100, 70, 9, 33)
    a, b = _run(c, True, schedule), _run(c, False, schedule)
    assert a[1] == b[1] == sum(schedule)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def test_graphs_of_8_steps_of_the_one_pass_update(monkeypatch):
    import test_gpu_graph_lengths as lengths
    make = lengths.make_gpu
    monkeypatch.setattr(lengths, "make_gpu", lambda c: make(c, passes=1))
    c = _case(40)
    schedule = (130, 25, 8, 3)
    a, b = _run(c, True, schedule), _run(c, False, schedule)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("dims,n", [((1025, 64, 96), 0), ((256, 257, 96), 300)])
def test_one_pass_mrt_in_thin_tiles(dims, n):
    c = mrt_case(dims, n)
    f1, x1 = run_passes(c, 4, 0)
    f2, x2 = run_passes(c, 4, 2)
    assert pop_error(f1, f2.astype(np.float64)) <= 2e-6
    assert n == 0 or np.abs(x1 - x2).max() <= 1e-6
