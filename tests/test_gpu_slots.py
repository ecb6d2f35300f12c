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


@pytest.mark.parametrize("n", [64, 1000])
def test_vertex_model_small_and_with_room_for_many_cells(n):
    # the same network in a context of its size and in one with room for many more
    # cells (empty cells and free vertices past the network)
    x, y, th, L = workloads.spv_uniform(n, 13)
    sims = [cg.AVM(n, L, L, x, y, th, v0=0.3, seed=3, t2_area=0.01, capacity=cap) for cap in (n, 40000)]
    for sim in sims:
        a0 = np.ones(sim.n)
        a0[:n // 10] = 0.0  # dying cells: triangles, T2s, empty cells
        sim.set_a0(a0)
    for steps in (1, 40):
        got = []
        for sim in sims:
            sim.step(steps)
            hx, hy, th_ = sim.state()
            vc, vn, cc, cv = sim.topology()
            A, P = sim.geometry()
            Fx, Fy, _ = sim.forces()
            got.append([t.cpu().numpy() for t in (hx[:2 * n], hy[:2 * n], th_[:n], vc[:2 * n], vn[:2 * n], cc[:n],
                                                  cv[:n], A[:n], P[:n], Fx[:2 * n], Fy[:2 * n])])
        for a, b in zip(*got):
            assert np.array_equal(a, b)
    c = [sim.counters() for sim in sims]
    assert c[0]["t1_total"] == c[1]["t1_total"] > 0 and c[0]["t2_total"] == c[1]["t2_total"]
    for sim in sims:
        sim.close()


def test_cocircular_cells_alone_and_inside_a_large_batch():
    # a square lattice: every quadruple is cocircular, so float values leave every slot open
    n, s = 400, 20
    k = np.arange(n)
    small = dict(n=n, Lx=float(s), Ly=float(s), p0=3.85, v0=1e-4), k % s + 0.5, k // s + 0.5, np.linspace(0.0, 6.0, n)
    big = _rep(LARGE, 12)
    alone = cg.SPV([small[0]], *small[1:], dt=0.002, seed=5)
    batch = cg.SPV([small[0], big[0]], *(np.concatenate([small[k], big[k]]) for k in (1, 2, 3)), dt=0.002, seed=5)
    for _ in range(4):
        alone.step(1)
        batch.step(1)
        for a, b in zip(alone.state() + alone.neighbors(), batch.state() + batch.neighbors()):
            assert np.array_equal(a.cpu().numpy(), b.cpu().numpy()[:n])
    assert alone.counters()["flagged_total"] > 0
    alone.close()
    batch.close()
