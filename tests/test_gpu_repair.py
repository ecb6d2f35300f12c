"""Rings of point sets at the edges of the ring search: more candidates than a
warp holds, cells whose neighbours lie many bins away, nearly coincident and
nearly collinear neighbours (exact decisions).  Bit-exact against the oracle."""
import numpy as np
import pytest

import oracle
import paper_1702_02939_gb300 as cg

pytestmark = pytest.mark.gpu


def _points(kind):
    rng = np.random.default_rng(3)
    if kind == "void":  # a hole of radius 5 spacings
        L, p = 40.0, rng.uniform(0.0, 40.0, (1600, 2))
        p = p[np.hypot(*(p - 20.0).T) > 5.0]
    elif kind == "dense":  # about 70 cells in the 25 bins around a cell of the patch
        L, p = 64.0, rng.uniform(0.0, 64.0, (4096, 2))
        patch = rng.uniform(10.0, 19.0, (150, 2))
        p = np.concatenate([p[~((p > 10.0) & (p < 19.0)).all(1)], patch, rng.uniform(10.0, 19.0, (70, 2))])
    elif kind == "pairs":  # every cell twice, 1e-5 to 1e-2 apart
        L, p = 32.0, rng.uniform(0.0, 32.0, (512, 2))
        r, a = 10.0 ** rng.uniform(-5.0, -2.0, 512), rng.uniform(0.0, 2.0 * np.pi, 512)
        p = np.concatenate([p, p + np.stack([r * np.cos(a), r * np.sin(a)], 1)]) % L
    else:  # rows of cells collinear to 1e-12
        L = 32.0
        p = np.stack([rng.uniform(0.0, L, 1024), np.repeat(np.arange(32), 32) + 0.5], 1)
        p[:, 1] += rng.uniform(-1e-12, 1e-12, 1024)
    return p[:, 0].copy(), p[:, 1].copy(), L


@pytest.mark.parametrize("kind", ["void", "dense", "pairs", "rows"])
def test_rings_equal_the_oracle(kind):
    x, y, L = _points(kind)
    n = len(x)
    Lx, Ly, _ = oracle.box(L)
    xs, ys = oracle.snap_positions(x, y, Lx, Ly)
    sim = cg.SPV([dict(n=n, Lx=L, Ly=L, p0=3.8, v0=0.05)], xs, ys, np.zeros(n))
    topo = oracle.triangulate(xs, ys, Lx, Ly)
    cnt, nbr = (t.cpu().numpy() for t in sim.neighbors())
    np.testing.assert_array_equal(cnt, topo.cnt)
    np.testing.assert_array_equal(nbr, topo.nbr)
    sim.close()


@pytest.mark.parametrize("n", [400, 4099])
def test_later_rounds_with_long_lists(n):
    """Moves of a fraction of a spacing: most cells are repaired, and the rounds
    after the first have many cells left."""
    rng = np.random.default_rng(5)
    L = float(np.sqrt(n))
    Lx, Ly, _ = oracle.box(L)
    xs, ys = oracle.snap_positions(rng.uniform(0.0, L, n), rng.uniform(0.0, L, n), Lx, Ly)
    sim = cg.SPV([dict(n=n, Lx=L, Ly=L, p0=3.8, v0=3.0)], xs, ys, rng.uniform(0.0, 6.28, n), KA=0.0, KP=0.0, dt=0.1,
                 seed=1, repair_cap=16)
    for _ in range(3):
        sim.step(1)
        x, y, _ = (t.cpu().numpy() for t in sim.state())
        topo = oracle.triangulate(x, y, Lx, Ly)
        cnt, nbr = (t.cpu().numpy() for t in sim.neighbors())
        np.testing.assert_array_equal(cnt, topo.cnt)
        np.testing.assert_array_equal(nbr, topo.nbr)
    c = sim.counters()
    assert c["repaired_total"] > c["flagged_total"] > n and c["loop_total"] > 3
    sim.close()
