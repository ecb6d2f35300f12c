"""The buffer of a checkpointed run: its size, and reverse passes repeated on it."""
import numpy as np
import pytest

import paper_1702_02939_gb300 as cg
import workloads

pytestmark = pytest.mark.gpu


def _sim(n):
    x, y, th, L = workloads.spv_uniform(n, 2)
    return cg.SPV([dict(n=n, Lx=L, Ly=L, p0=3.8, v0=0.1)], x, y, th, dt=0.002, seed=1)


def test_one_saved_state_per_checkpoint_and_one_segment():
    sim = _sim(301)
    size = lambda nsteps, every: cg.cg_backward_bytes(sim.ctx, nsteps, every)
    state = size(30, 10) - size(20, 10)
    for nsteps, every in ((50, 50), (5, 50), (50, 10), (51, 10), (1, 7)):
        states = -(-nsteps // every) + 1 + every
        assert size(nsteps, every) - size(1, 1) == (states - 3) * state
    sim.close()


@pytest.mark.parametrize("every", [12, 5, 6, 1])  # one segment, a short last one, full ones, one step each
def test_reverse_passes_repeated_on_one_buffer(every):
    n, steps = 301, 12
    rng = np.random.default_rng(3)
    g = [rng.standard_normal(n) for _ in range(4)]
    got = []
    sim = _sim(n)
    x, y, th = sim.state()
    for k in (every, steps):  # steps: one segment, nothing recomputed
        sim.set_state(x, y, th)
        sim.set_step(0)
        bw = sim.run_checkpointed(steps, k)
        for _ in range(3):
            out = sim.backward(bw, steps, k, *g)
            got.append([t.cpu().numpy() for t in out[:4]] + [np.array(out[4:])])
    sim.close()
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert np.array_equal(a, b)
