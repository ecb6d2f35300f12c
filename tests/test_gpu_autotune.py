"""The trials of the autotuner time steps alone."""
import pytest

import paper_1702_02939_gb300 as cg
import workloads

pytestmark = pytest.mark.gpu


def test_a_shape_tried_late_is_timed_as_the_first():
    """A grid of one block per SM for the circumcircle test costs about 10 us a
    step; its field is tried after several others.  Trials that also build a
    graph of several steps (200 us, 20 us a step) would keep it."""
    n = 40000
    x, y, th, L = workloads.spv_uniform(n, 1)
    sim = cg.SPV([dict(n=n, Lx=L, Ly=L, p0=3.8, v0=0.1)], x, y, th, dt=0.005, seed=1)
    sim.step(50)
    sim.set_launch(test_blocks_per_sm=1)
    best, ms = sim.autotune(10)
    assert best["test_blocks_per_sm"] != 1
    sim.close()
