"""Vertex positions handed in outside [0, L): areas, perimeters, forces and the
next step are those of the same network inside the box."""
import numpy as np
import pytest

import oracle
import paper_1702_02939_gb300 as cg
import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [64, 100])  # sides 8 (a power of two) and 10
@pytest.mark.parametrize("where", ["upper side", "one box up", "one box down", "mixed", "three boxes up", "zero minus"])
def test_positions_outside_the_box(n, where):
    x, y, th, L = workloads.spv_uniform(n, 5)
    Lx, Ly, _ = oracle.box(L)
    net = oracle.avm_build(*oracle.snap_positions(x, y, Lx, Ly), Lx, Ly)
    # a vertex on each lower side, all positions multiples of 2^-40: shifts by
    # whole boxes are exact
    grid = 2.0 ** -40
    hx, hy = (np.rint(((h - h[k]) % s) / grid) * grid % s for h, k, s in ((net.hx, 0, Lx), (net.hy, 7, Ly)))
    assert hx[0] == 0.0 and hy[7] == 0.0
    rng = np.random.default_rng(1)
    few = rng.random(2 * n) < 0.2
    k = {"upper side": (hx == 0.0) | (hy == 0.0), "one box up": few, "one box down": -1 * few,
         "mixed": rng.integers(-2, 3, 2 * n), "three boxes up": np.full(2 * n, 3), "zero minus": np.zeros(2 * n)}[where]
    gx, gy = (h + k * s for h, s in ((hx, Lx), (hy, Ly)))
    if where == "upper side":
        gx, gy = np.where(hx == 0.0, Lx, hx), np.where(hy == 0.0, Ly, hy)
    if where == "zero minus":
        gx, gy = np.where(hx == 0.0, -0.0, hx), np.where(hy == 0.0, -1e-300, hy)
    got = []
    for a, b in ((hx, hy), (gx, gy)):
        sim = cg.AVM(n, L, L, x, y, th, v0=0.3, t1_threshold=0.0, seed=3)
        sim.set_state(a, b, th, net.vc, net.vn, net.cc, net.cv)
        sx, sy, _ = (t.cpu().numpy() for t in sim.state())
        assert np.array_equal(sx, hx) and np.array_equal(sy, hy)  # reduced into the box
        out = [t.cpu().numpy() for t in (*sim.geometry(), *sim.forces()[:2])]
        sim.step(1)
        got.append((out, [t.cpu().numpy() for t in sim.state()[:2]]))
        sim.close()
    for a, b in zip(got[0][0] + got[0][1], got[1][0] + got[1][1]):
        assert np.array_equal(a, b)
    oFx, oFy, oA, oP, _ = oracle.avm_forces(oracle.AvmNet(n, Lx, Ly, hx, hy, net.vc, net.vn, net.cc, net.cv), 3.8)
    scale = max(np.abs(oFx).max(), np.abs(oFy).max())
    for a, b, s in zip(got[1][0], (oA, oP, oFx, oFy), (1.0, 1.0, scale, scale)):
        assert np.abs(a - b).max() <= 1e-10 * max(s, np.abs(b).max())
