"""Kernels with one thread per (cell, ring slot), which small systems and the
lists of a step take, against the kernels with one thread per cell, which large
ones take: a system gives the same bits alone and inside a batch too large for
the slot kernels."""
import numpy as np
import pytest

import paper_1702_02939_gb300 as cg
import workloads

pytestmark = pytest.mark.gpu

LARGE = 160000  # more cells than any slot kernel takes


def _rep(n, seed, p0=3.85, v0=0.1):
    x, y, th, L = workloads.spv_uniform(n, seed)
    return dict(n=n, Lx=L, Ly=L, p0=p0, v0=v0), x, y, th


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("n", [64, 95, 97, 1000, 4099])  # below, at and past whole blocks of 32 cells
def test_small_system_alone_and_inside_a_large_batch(n, precision):
    # uniform random cells: rings of 3 to more than 8 neighbours
    small, big = _rep(n, 11), _rep(LARGE, 12)
    reps = [small[0], big[0]]
    xs, ys, ths = (np.concatenate([small[k], big[k]]) for k in (1, 2, 3))
    alone = cg.SPV(reps[:1], *small[1:], dt=0.002, seed=5, precision=precision)
    batch = cg.SPV(reps, xs, ys, ths, dt=0.002, seed=5, precision=precision)
    assert int(batch.neighbors()[0].max()) > 8
    for steps in (0, 1, 3):
        alone.step(steps)
        batch.step(steps)
        got = [t.cpu().numpy() for t in (*alone.state(), *alone.geometry(), *alone.forces()[:2])]
        ref = [t.cpu().numpy()[:n] for t in (*batch.state(), *batch.geometry(), *batch.forces()[:2])]
        for a, b in zip(got, ref):
            assert np.array_equal(a, b)
        assert np.array_equal(alone.neighbors()[1].cpu().numpy(), batch.neighbors()[1].cpu().numpy()[:n])
    alone.close()
    batch.close()
