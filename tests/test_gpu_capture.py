"""Graphs of several steps are built for long runs only, where they pay."""
import time

import numpy as np
import pytest

import paper_1702_02939_gb300 as cg
import workloads

pytestmark = pytest.mark.gpu


def test_a_few_steps_between_changes_of_the_moduli():
    """Ten steps per value of K_A cost no more in one call than in ten: neither
    builds a graph of several steps after each change."""
    n = 1024
    x, y, th, L = workloads.spv_uniform(n, 1)
    sims = [cg.SPV([dict(n=n, Lx=L, Ly=L, p0=3.8, v0=0.1)], x, y, th, dt=0.005, seed=1) for _ in range(2)]
    times = [[], []]
    for sim in sims:
        sim.step(200)  # a long run already
        sim.sync()
    for k in range(30):
        for sim, calls, out in zip(sims, (1, 10), times):
            t0 = time.perf_counter()
            sim.set_moduli(1.0 + 1e-3 * k, 1.0)
            for _ in range(calls):
                sim.step(10 // calls)
            sim.sync()
            out.append(time.perf_counter() - t0)
    assert np.median(times[0]) < 1.3 * np.median(times[1])
    for a, b in zip(*(sim.state() for sim in sims)):
        assert bool((a == b).all())
    for sim in sims:
        sim.close()


def test_long_runs_after_a_change_of_the_moduli():
    """Past 64 steps with the same moduli a call's steps go several per launch
    again; the result is that of one call per step."""
    n = 150
    x, y, th, L = workloads.spv_uniform(n, 6)
    got = []
    for single in (False, True):
        sim = cg.SPV([dict(n=n, Lx=L, Ly=L, p0=3.8, v0=0.2)], x, y, th, seed=3)
        for KA, steps in ((1.0, 90), (1.5, 70), (1.5, 33), (1.2, 17)):
            sim.set_moduli(KA, 0.5)
            for _ in range(steps if single else 1):
                sim.step(1 if single else steps)
        got.append([t.cpu().numpy() for t in sim.state()])
        sim.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
