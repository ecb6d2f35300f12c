"""Forces of cells with near and far polygon vertices (a small cluster of cells
in an otherwise sparse box), against extended precision: every vertex, edge and
area term counts as FP64 would hold it for itself, however far the cell's other
vertices are."""
import numpy as np
import pytest

import oracle
import paper_1702_02939_gb300 as cg
import workloads

pytestmark = pytest.mark.gpu

LD = np.longdouble
U = 2.0 ** -53
KA, KP, P0 = 0.5, 1.0, 3.8


def _cross(a, b):
    return a[0] * b[1] - a[1] * b[0]


def _reference(x, y, L, cnt, nbr):
    """Forces in extended precision, and what FP64 may be off by when a
    circumcentre carries 4 roundings and the squared lengths it is made of are
    cut to 61 bits, and an edge, a cell's area and perimeter and their sums carry
    the errors of the vertices they are made of and 8 roundings of their own."""
    n = len(x)
    pos = [np.array([LD(x[i]), LD(y[i])]) for i in range(n)]
    half, box = LD(L) / 2, LD(L)

    def off(i, j):
        d = pos[j] - pos[i]
        return np.where(d > half, d - box, np.where(d < -half, d + box, d))

    ring = [list(nbr[i][:cnt[i]]) for i in range(n)]
    cell = []  # per cell: circumcentres, determinants, offsets, dE/dh and its error per vertex
    for i in range(n):
        r = [off(i, j) for j in ring[i]]
        m = len(r)
        h, det, dh = [], [], []
        for a in range(m):
            p, q = r[a], r[(a + 1) % m]
            D = _cross(p, q)
            lp, lq = p @ p, q @ q
            h.append(np.array([q[1] * lp - p[1] * lq, p[0] * lq - q[0] * lp]) / (2 * D))
            det.append(D)
            cut = 2.0 ** -61 * max(lp, lq) * (np.sqrt(lp) + np.sqrt(lq)) / (2 * D)
            dh.append(4 * U * np.sqrt(h[-1] @ h[-1]) + cut)
        size = [np.sqrt(v @ v) for v in h]
        e, err, length = [], [], []  # edge ending at a
        for a in range(m):
            d = h[a] - h[a - 1]
            s = np.sqrt(d @ d)
            e.append(d / s)
            length.append(s)
            err.append(2 * (dh[a] + dh[a - 1]) / s + 8 * U)
        A = sum(_cross(h[a - 1], h[a]) for a in range(m)) / 2
        P = sum(length)
        dA = sum(size[a - 1] * dh[a] + dh[a - 1] * size[a] + 8 * U * size[a - 1] * size[a] for a in range(m))
        dP = sum(err[a] * length[a] for a in range(m)) + 8 * U * P
        ka, kp = 2 * KA * (A - 1), 2 * KP * (P - P0)
        dka, dkp = 2 * KA * dA + 8 * U * abs(ka), 2 * KP * (dP + 2 * U * P0) + 8 * U * abs(kp)
        g, dg = [], []
        for a in range(m):
            b = (a + 1) % m
            t = h[b] - h[a - 1]
            gA = np.array([t[1], -t[0]]) / 2
            gP = e[a] - e[b]
            sA, sP = np.sqrt(gA @ gA), np.sqrt(gP @ gP)
            g.append(ka * gA + kp * gP)
            dg.append(dka * sA + abs(ka) * (dh[b] + dh[a - 1] + 8 * U * sA) + dkp * sP +
                      abs(kp) * (err[a] + err[b] + 8 * U * sP))
        cell.append((h, det, r, g, dg, dh))
    F, B = np.zeros((n, 2), LD), np.zeros((n, 2))
    for i in range(n):
        h, det, r, _, _, dh = cell[i]
        m = len(h)
        for a in range(m):
            j, k = ring[i][a], ring[i][(a + 1) % m]
            G, dG = cell[i][3][a].copy(), cell[i][4][a]
            for c, first in ((j, k), (k, i)):  # the triangle's slot around j starts at k, around k at i
                s = ring[c].index(first)
                G += cell[c][3][s]
                dG += cell[c][4][s]
            q, p = r[(a + 1) % m], r[a]
            w = np.array([q[1] - p[1], p[0] - q[0]])
            F[i] -= h[a] / det[a] * (w @ G)
            sw, sG = np.sqrt(w @ w), np.sqrt(G @ G)
            B[i] += (np.abs(h[a]).astype(float) * float(sw * (dG + 16 * U * sG)) + float(dh[a] * sw * sG)) / float(det[a])
    return F, B + 8 * U * np.abs(F).astype(float)


@pytest.mark.parametrize("eps", [2.0 ** -k for k in (4, 8, 12, 16)])
def test_forces_of_cells_with_a_far_vertex(eps):
    L = 8.0
    rng = np.random.default_rng(4)
    x, y = rng.uniform(0.0, L, (2, 60))
    keep = np.hypot(x - 3.1, y - 4.3) > 0.5
    r, a = eps * np.sqrt(rng.uniform(0.0, 1.0, 9)), rng.uniform(0.0, 2.0 * np.pi, 9)
    x, y = np.concatenate([x[keep], 3.1 + r * np.cos(a)]), np.concatenate([y[keep], 4.3 + r * np.sin(a)])
    n = len(x)
    Lx, Ly, _ = oracle.box(L)
    xs, ys = oracle.snap_positions(x, y, Lx, Ly)
    topo = oracle.triangulate(xs, ys, Lx, Ly)
    F, B = _reference(xs, ys, L, topo.cnt, topo.nbr.reshape(n, -1))
    small = dict(n=n, Lx=L, Ly=L, p0=P0, v0=0.1)
    sim = cg.SPV([small], xs, ys, np.zeros(n), KA=KA, KP=KP)
    got = [t.cpu().numpy() for t in sim.forces()[:2]]
    sim.close()
    for k in range(2):
        assert (np.abs((got[k] - F[:, k]).astype(float)) <= B[:, k]).all()
    # inside a batch too large for the kernel with a thread per slot: the same bits
    bx, by, bth, bL = workloads.spv_uniform(160000, 12)
    sim = cg.SPV([small, dict(n=160000, Lx=bL, Ly=bL, p0=P0, v0=0.1)], np.concatenate([xs, bx]),
                 np.concatenate([ys, by]), np.zeros(n + 160000), KA=KA, KP=KP)
    for a, b in zip(got, sim.forces()[:2]):
        assert np.array_equal(a, b.cpu().numpy()[:n])
    sim.close()
