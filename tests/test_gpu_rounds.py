"""Repair rounds that find most cells flagged, at the sizes where they go from one
cluster to the grid: rings bit-exact against the oracle, and no size at which
such a step takes much longer than the next larger one that uses the grid."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1702_02939_gb300 as cg

pytestmark = pytest.mark.gpu


def _driven(n, precision="f64"):
    """Moves of 0.3 of a spacing a step."""
    rng = np.random.default_rng(5)
    L = float(np.sqrt(n))
    Lx, Ly, _ = oracle.box(L)
    xs, ys = oracle.snap_positions(rng.uniform(0.0, L, n), rng.uniform(0.0, L, n), Lx, Ly)
    sim = cg.SPV([dict(n=n, Lx=L, Ly=L, p0=3.8, v0=3.0)], xs, ys, rng.uniform(0.0, 6.28, n), KA=0.0, KP=0.0, dt=0.1,
                 seed=1, repair_cap=16, precision=precision)
    return sim, Lx, Ly


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("n", [1024, 1025, 4096, 4097])
def test_rings_at_the_lines_between_cluster_and_grid(n, precision):
    sim, Lx, Ly = _driven(n, precision)
    for _ in range(3):
        sim.step(1)
        x, y, _ = (t.cpu().numpy() for t in sim.state())
        topo = oracle.triangulate(x, y, Lx, Ly)
        cnt, nbr = (t.cpu().numpy() for t in sim.neighbors())
        np.testing.assert_array_equal(cnt, topo.cnt)
        np.testing.assert_array_equal(nbr, topo.nbr)
    c = sim.counters()
    assert c["repaired_total"] > c["flagged_total"] > 2.5 * n and c["loop_total"] > 3
    sim.close()


def test_rounds_counted_alike():
    """A step without a flagged cell counts one round and no repair."""
    x, y = (v.ravel() + 0.01 for v in np.meshgrid(np.arange(48.0), np.arange(48.0)))
    for n in (961, 2209):  # cluster alone, grid repair and cluster
        m = int(np.sqrt(n))
        keep = (x < m) & (y < m)
        xs, ys = x[keep] + 0.3 * (y[keep] // 1 % 2), y[keep]
        sim = cg.SPV([dict(n=n, Lx=float(m), Ly=float(m), p0=3.8, v0=0.0)], xs, ys, np.zeros(n), KA=0.0, KP=0.0, seed=1)
        c0 = sim.counters()
        sim.step(5)
        c = sim.counters()
        assert c["loop_total"] - c0["loop_total"] == 5 and c["flagged_total"] == c0["flagged_total"]
        assert c["repaired_total"] == c0["repaired_total"]
        sim.close()


def test_a_step_that_repairs_every_cell_takes_the_chip():
    def ms(n):
        sim, _, _ = _driven(n)
        out = []
        for _ in range(17):
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            sim.step(1)
            b.record()
            torch.cuda.synchronize()
            out.append(a.elapsed_time(b))
        sim.close()
        return float(np.median(out[1:]))

    assert ms(4096) < 2.0 * ms(4160)
