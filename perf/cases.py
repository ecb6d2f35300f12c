"""Performance cases of the framework: what a program that simulates tissues
with it calls, over the sizes it is called at.

Every case goes through the public classes and functions of the package.  The
inputs are tissues at unit density: a triangular arrangement of cells in a
periodic square box with Gaussian positional disorder (and a few vacancies
where the number of cells does not fill the arrangement), directors uniform in
[0, 2 pi), the model parameters of the paper's runs (p0 about 3.8, v0 0.01 to
0.5, dt 0.01).  `exact` repeats a pass in plain torch and numpy in 64 bits:
Delaunay rings by gift wrapping over a cell grid, the energy of Eq. 1 from the
circumcentres, forces by automatic differentiation, the Philox director noise,
and for the vertex model the T1 passes edge by edge.
"""
import math

import numpy as np
import torch

import paper_1702_02939_gb300 as cg

DEV = "cuda"
F64 = torch.float64
RING = 16
DT, DR = 0.01, 1.0
T1_THRESHOLD = 0.04
DISORDER = 0.16  # standard deviation of the positions, in mean spacings

SPV = dict(kind="spv", precision="f64", p0=3.85, v0=0.1)


def listed():
    return [
        # a small tissue followed in time, one saved configuration per pass:
        # parameter studies run thousands of these, bound by launches and latency
        dict(SPV, name="spv_1k", n=1024, steps=10),
        # the size of most published runs, in the fluid regime
        dict(SPV, name="spv_16k", n=16384, steps=10),
        # the benchmark's tissue
        dict(SPV, name="spv_256k", n=262144, steps=5),
        # a large solid tissue with a ragged number of cells: few neighbour changes
        dict(SPV, name="spv_1m_solid", n=1000003, steps=3, p0=3.8, v0=0.01),
        # the benchmark's tissue in single precision
        dict(SPV, name="spv_256k_f32", n=262144, steps=5, precision="f32"),
        # an ensemble of independent tissues of mixed sizes advanced together
        dict(kind="batch", name="spv_batch", replicas=128, n_min=256, n_max=16384, steps=5),
        # a tissue driven from the host: speeds in and positions out every step
        dict(SPV, name="spv_256k_io", kind="io", n=262144, steps=4),
        # one configuration from elsewhere evaluated: neighbours, areas,
        # perimeters, forces and energy
        dict(SPV, name="spv_64k_eval", kind="eval", n=65536),
        # a differentiable run (inverse problems): forward, loss and gradients
        dict(SPV, name="spv_4k_grad", kind="grad", n=4096, steps=12, every=6),
        # the neighbours of a point set alone, without device allocation
        dict(kind="neighbours", name="neighbours_2k", n=2000),
        # the vertex model, small and at the benchmark's size
        dict(kind="avm", name="avm_4k", n=4096, steps=20, sort_every=0, dying=0),
        dict(kind="avm", name="avm_64k", n=65536, steps=10, sort_every=100, dying=0),
    ]


def _log_size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spv", "spv", "spv", "batch", "io", "eval", "grad", "neighbours", "avm", "avm"])
    p0, v0 = round(rng.uniform(3.6, 3.9), 4), round(math.exp(rng.uniform(math.log(0.01), math.log(0.3))), 4)
    if kind == "spv":
        return dict(kind=kind, precision=rng.choice(["f64", "f64", "f32"]), n=_log_size(rng, 256, 1000000),
                    steps=rng.randint(1, 3), p0=p0, v0=v0)
    if kind == "batch":
        return dict(kind=kind, replicas=rng.randint(2, 128), n_min=256, n_max=_log_size(rng, 512, 16384),
                    steps=rng.randint(1, 5))
    if kind == "io":
        return dict(kind=kind, precision="f64", n=_log_size(rng, 1000, 262144), steps=rng.randint(1, 4), p0=p0, v0=v0)
    if kind == "eval":
        return dict(kind=kind, precision="f64", n=_log_size(rng, 256, 262144), p0=p0, v0=v0)
    if kind == "grad":
        return dict(kind=kind, precision="f64", n=_log_size(rng, 400, 16384), steps=rng.randint(2, 20),
                    every=rng.randint(2, 10), p0=p0, v0=v0)
    if kind == "neighbours":
        return dict(kind=kind, n=_log_size(rng, 64, 16384))
    return dict(kind=kind, n=_log_size(rng, 400, 262144), steps=rng.randint(1, 10),
                sort_every=rng.choice([0, 100]), dying=rng.choice([0, 0, 1]))


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _tissue(n, gen):
    """(x, y, theta, L) of n cells at unit density."""
    L = math.sqrt(n)
    rows = 2 * max(2, math.ceil(0.5 * math.sqrt(n * 2.0 / math.sqrt(3.0))))
    cols = math.ceil(n / rows)
    keep = torch.randperm(rows * cols, generator=gen, device=DEV)[:n].sort().values
    r, c = keep // cols, keep % cols
    jit = DISORDER * torch.randn(2, n, generator=gen, device=DEV, dtype=F64)
    x = (c.to(F64) + 0.5 * (r % 2) + 0.25) * (L / cols) + jit[0]
    y = (r.to(F64) + 0.5) * (L / rows) + jit[1]
    theta = 2.0 * math.pi * torch.rand(n, generator=gen, device=DEV, dtype=F64)
    return torch.remainder(x, L), torch.remainder(y, L), theta, L


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _sizes(case):
    """Sizes of the ensemble's tissues, log-uniform."""
    lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
    return np.rint(np.exp(np.random.default_rng(7).uniform(lo, hi, case["replicas"]))).astype(int)


def _replicas(case, seed):
    """p0 uniform on [3.6, 4.0), v0 uniform on [0.01, 0.5)."""
    n = _sizes(case)
    rng = np.random.default_rng(seed)
    p0, v0 = rng.uniform(3.6, 4.0, len(n)), rng.uniform(0.01, 0.5, len(n))
    gen = _gen(seed)
    parts = [_tissue(int(k), gen) for k in n]
    reps = [dict(n=int(n[r]), Lx=parts[r][3], Ly=parts[r][3], p0=float(p0[r]), v0=float(v0[r]))
            for r in range(len(n))]
    return reps, [torch.cat([p[k] for p in parts]) for k in range(3)]


def _inputs(case, seed):
    """Everything a case takes from its seed."""
    if case["kind"] == "batch":
        reps, (x, y, theta) = _replicas(case, seed)
        return dict(reps=reps, x=x, y=y, theta=theta)
    gen = _gen(seed)
    x, y, theta, L = _tissue(case["n"], gen)
    d = dict(x=x, y=y, theta=theta, L=L)
    if "p0" in case:
        d["reps"] = [dict(n=case["n"], Lx=L, Ly=L, p0=case["p0"], v0=case["v0"])]
    if case["kind"] == "io":  # speeds that vary from cell to cell and from step to step
        u = torch.rand(case["steps"], case["n"], generator=gen, device=DEV, dtype=F64)
        d["v0"] = case["v0"] * (0.5 + u)
    if case["kind"] == "grad":
        d["p0"] = case["p0"] + 0.2 * torch.rand(case["n"], generator=gen, device=DEV, dtype=F64) - 0.1
    if case["kind"] == "avm" and case["dying"]:  # one cell in a hundred shrinks and is removed
        d["a0"] = (torch.rand(case["n"], generator=gen, device=DEV, dtype=F64) > 0.01).to(F64)
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    s = dict(case=case)
    kind = case["kind"]
    if kind == "neighbours":
        n = case["n"]
        s.update(x=d["x"], y=d["y"], L=d["L"], cnt=torch.empty(n, dtype=torch.int32, device=DEV),
                 nbr=torch.empty(n, RING, dtype=torch.int32, device=DEV),
                 stream=torch.cuda.current_stream().cuda_stream)
        return s
    if kind == "avm":
        s["sim"] = cg.AVM(case["n"], d["L"], d["L"], d["x"], d["y"], d["theta"], p0=3.8, v0=0.1, dt=DT, Dr=DR,
                          t1_threshold=T1_THRESHOLD, t2_area=0.01 if case["dying"] else 0.0, seed=int(seed),
                          sort_every=case["sort_every"], device=DEV)
        if case["dying"]:
            s["sim"].set_a0(d["a0"])
        return s
    s["sim"] = cg.SPV(d["reps"], d["x"], d["y"], d["theta"], dt=DT, Dr=DR, seed=int(seed),
                      precision=case.get("precision", "f64"), device=DEV)
    if kind == "io":
        s["v0"] = d["v0"].cpu().pin_memory()
        s["xy"] = torch.empty(2, case["steps"], case["n"], dtype=F64).pin_memory()
    if kind == "eval":  # configurations arrive from elsewhere, another one each pass
        gen = _gen(seed + 1)
        s["next"] = [(d["x"], d["y"])] + [_tissue(case["n"], gen)[:2] for _ in range(2)]
        s["k"] = 0
    if kind == "grad":
        s.update(d)
    return s


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def _loss(A, P):
    """Deviation of the shape index from 3.95 (mean over cells)."""
    return ((A * (P / torch.sqrt(A) - 3.95)) ** 2).mean()


def run(s):
    case = s["case"]
    kind, sim = case["kind"], s.get("sim")
    if kind in ("spv", "batch"):
        sim.step(case["steps"])
        return sim.state()
    if kind == "io":
        sim.run_io(case["steps"], v0=s["v0"], x=s["xy"][0], y=s["xy"][1], v0_stride=case["n"], out_stride=case["n"])
        return s["xy"]
    if kind == "eval":
        x, y = s["next"][s["k"] % len(s["next"])]
        s["k"] += 1
        sim.set_state(x, y)
        cnt, nbr = sim.neighbors()
        A, P = sim.geometry()
        Fx, Fy, E = sim.forces()
        return cnt, nbr, A, P, Fx, Fy, E
    if kind == "grad":
        leaf = [s["x"].clone(), s["y"].clone(), s["p0"].clone()] + [torch.tensor(v, dtype=F64)
                                                                    for v in (case["v0"], 1.0, 1.0)]
        for t in leaf:
            t.requires_grad_(True)
        x, y, A, P = cg.spv_run_differentiable(sim, *leaf, s["theta"], case["steps"], ckpt_every=case["every"])
        loss = _loss(A, P)
        loss.backward()
        return [x.detach(), y.detach(), A.detach(), P.detach(), loss.detach()] + [t.grad for t in leaf]
    if kind == "neighbours":
        cg.cg_triangulate_noalloc(case["n"], s["L"], s["L"], s["x"], s["y"], s["cnt"], s["nbr"], s["stream"])
        return s["cnt"], s["nbr"]
    sim.step(case["steps"])
    return list(sim.state()) + list(sim.topology())


def _cells(case):
    if case["kind"] != "batch":
        return case["n"]
    return int(_sizes(case).sum())


def work(case):
    """Per cell: the model's state (positions, director, parameters, ring)
    read and written once a step; the arithmetic of the method a step (six
    neighbours a cell; each circumcentre once)."""
    n, kind, k = _cells(case), case["kind"], case.get("steps", 1)
    if kind in ("spv", "batch"):
        return {"bytes": n * (84.0 * k + 24), "flops": 390.0 * n * k}
    if kind == "io":
        return {"bytes": n * (84.0 + 24) * k, "flops": 390.0 * n * k}
    if kind == "eval":  # positions in; rings, A, P and forces out
        return {"bytes": n * (16.0 + 68 + 16 + 16 + 8), "flops": 350.0 * n}
    if kind == "grad":  # forward, and the tangent of every step (twice its arithmetic)
        return {"bytes": n * (84.0 + 120.0) * k, "flops": 390.0 * n * k * 3}
    if kind == "neighbours":
        return {"bytes": n * (16.0 + 68), "flops": 60.0 * n}
    # vertex model: 2 vertices a cell; state and topology out once a pass
    return {"bytes": n * (150.0 * k + 40 + 116), "flops": 240.0 * n * k}


# --------------------------------------------------------------------------
# the same passes in plain torch and numpy, 64 bits
# --------------------------------------------------------------------------
def _image(d, L):
    return d - L * torch.round(d / L)


def _offsets(x, y, L, idx):
    """Minimum-image offsets of the cells idx (or -1) from each row's cell."""
    j = idx.clamp(min=0)
    return _image(x[j] - x[:, None], L), _image(y[j] - y[:, None], L)


def _wrap(px, py, me, cand):
    """Rings of some cells by gift wrapping over their candidates (cell
    indices, -1 unused; offsets px, py): [rows, RING] cell indices and the
    largest squared circumradius of each."""
    bad = (cand < 0) | (cand == me[:, None])
    l2 = torch.where(bad, math.inf, px * px + py * py)
    rows = torch.arange(len(me), device=me.device)
    first = l2.argmin(1)
    g = first
    ring = torch.full((len(me), RING), -1, dtype=torch.int64, device=me.device)
    open_ = torch.ones(len(me), dtype=torch.bool, device=me.device)
    r2 = torch.zeros(len(me), dtype=F64, device=me.device)
    for a in range(RING):
        ring[:, a] = torch.where(open_, cand[rows, g], -1)
        gx, gy = px[rows, g][:, None], py[rows, g][:, None]
        cr = gx * py - gy * px
        s = torch.where(bad | (cr <= 0), math.inf, (l2 - gx * px - gy * py) / cr)
        s[rows, g] = math.inf
        t, nxt = s.min(1)
        r = 0.25 * (gx[:, 0] ** 2 + gy[:, 0] ** 2) * (1 + t * t)
        r2 = torch.where(open_, torch.maximum(r2, r), r2)
        open_ = open_ & (nxt != first)
        g = torch.where(open_, nxt, g)
        if not bool(open_.any()):
            return ring, r2
    raise RuntimeError("a ring did not close")


def _delaunay(x, y, L):
    """Delaunay rings [n, RING] (counter-clockwise, -1 past the end)."""
    n = len(x)
    x, y = x.detach(), y.detach()
    nb = max(5, int(L))
    w = L / nb
    bx, by = (x / w).long().clamp(max=nb - 1), (y / w).long().clamp(max=nb - 1)
    b = by * nb + bx
    order = b.argsort()
    count = torch.bincount(b, minlength=nb * nb)
    start = count.cumsum(0) - count
    ring = torch.empty(n, RING, dtype=torch.int64, device=x.device)
    todo = torch.arange(n, device=x.device)
    half = 2
    while len(todo):
        half = min(half, (nb - 1) // 2)
        side = torch.arange(-half, half + 1, device=x.device)
        later = []
        for part in todo.split(1 << 17):
            cb = (((by[part, None] + side) % nb)[:, :, None] * nb + ((bx[part, None] + side) % nb)[:, None, :]).flatten(1)
            most = int(count[cb].max())
            k = torch.arange(most, device=x.device)
            at = (start[cb][:, :, None] + k).clamp(max=n - 1)
            cand = torch.where(k < count[cb][:, :, None], order[at], -1).flatten(1)
            j = cand.clamp(min=0)
            px, py = _image(x[j] - x[part, None], L), _image(y[j] - y[part, None], L)
            ring[part], r2 = _wrap(px, py, part, cand)
            if half < (nb - 1) // 2:  # unseen cells are farther than half * w
                later.append(part[~(4.0 * r2 < (half * w) ** 2)])
        todo = torch.cat(later) if later else todo[:0]
        half *= 2
    return ring


def _next(ring, cnt):
    """Index of the following slot in each ring."""
    a = torch.arange(RING, device=ring.device).expand_as(ring)
    return torch.where(a + 1 < cnt[:, None], a + 1, 0)


def _spv_geometry(x, y, L, ring):
    """Areas and perimeters from the circumcentres (x, y, L per cell)."""
    used = ring >= 0
    cnt = used.sum(1)
    j = torch.where(used, ring, ring[:, :1])
    Lc = L[:, None]
    ax, ay = _image(x[j] - x[:, None], Lc), _image(y[j] - y[:, None], Lc)
    nx = _next(ring, cnt)
    bx, by = ax.gather(1, nx), ay.gather(1, nx)
    det = 2.0 * (ax * by - ay * bx)
    det = torch.where(used, det, 1.0)
    la, lb = ax * ax + ay * ay, bx * bx + by * by
    hx, hy = (by * la - ay * lb) / det, (ax * lb - bx * la) / det
    kx, ky = hx.gather(1, nx), hy.gather(1, nx)
    A = 0.5 * torch.where(used, hx * ky - kx * hy, 0.0).sum(1)
    e2 = torch.where(used, (kx - hx) ** 2 + (ky - hy) ** 2, 1.0)
    P = torch.where(used, torch.sqrt(e2), 0.0).sum(1)
    return A, P


def _philox(tag, step, seed):
    """Philox4x32-10 words of the counters (tag, step, 0)."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [tag.astype(np.uint64), np.full(len(tag), step & 0xFFFFFFFF, np.uint64),
         np.full(len(tag), step >> 32, np.uint64), np.zeros(len(tag), np.uint64)]
    k = [seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF]
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k[0]), p1 & m32,
             (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k[1]), p0 & m32]
        k = [(k[0] + 0x9E3779B9) & 0xFFFFFFFF, (k[1] + 0xBB67AE85) & 0xFFFFFFFF]
    return c


def _noise(n, step, seed, precision="f64"):
    """One standard normal per cell (Box-Muller, cosine branch)."""
    r = _philox(np.arange(n), step, seed)
    if precision == "f32":  # uniforms of 24 bits
        u1, u2 = (((w >> np.uint64(8)) + np.uint64(1)).astype(np.float64) * 2.0 ** -24 for w in (r[0], r[2]))
    else:
        u1, u2 = (((((a << np.uint64(32)) | b) >> np.uint64(11)) + np.uint64(1)).astype(np.float64) * 2.0 ** -53
                  for a, b in ((r[0], r[1]), (r[2], r[3])))
    return torch.from_numpy(np.sqrt(-2.0 * np.log(u1)) * np.cos(2.0 * np.pi * u2)).to(DEV)


def _per_cell(reps, field):
    return torch.cat([torch.full((r["n"],), float(r[field]), dtype=F64, device=DEV) for r in reps])


def _rings(x, y, reps):
    out, at = [], 0
    for r in reps:
        sl = slice(at, at + r["n"])
        ring = _delaunay(x[sl], y[sl], r["Lx"])
        out.append(torch.where(ring >= 0, ring + at, -1))
        at += r["n"]
    return torch.cat(out)


def _spv_energy(x, y, L, ring, p0, KA=1.0, KP=1.0):
    A, P = _spv_geometry(x, y, L, ring)
    return A, P, (KA * (A - 1.0) ** 2 + KP * (P - p0) ** 2).sum()


def _spv_step(x, y, theta, reps, L, p0, v0, KA=1.0, KP=1.0, grad=False):
    """Positions after one step of Eq. 3; differentiable when `grad`."""
    ring = _rings(x, y, reps)
    if not grad:
        x, y = x.detach().requires_grad_(True), y.detach().requires_grad_(True)
    E = _spv_energy(x, y, L, ring, p0, KA, KP)[2]
    gx, gy = torch.autograd.grad(E, (x, y), create_graph=grad)
    x, y = x + DT * (v0 * torch.cos(theta) - gx), y + DT * (v0 * torch.sin(theta) - gy)
    if not grad:
        x, y = x.detach(), y.detach()
    return x - L * torch.floor(x.detach() / L), y - L * torch.floor(y.detach() / L)


def exact(case, seed):
    kind = case["kind"]
    if kind == "avm" and case["dying"]:
        return None  # removals of cells are not written out here
    d = _inputs(case, seed)
    if kind == "avm":
        return _exact_avm(case, seed, d)
    x, y, theta = d["x"], d["y"], d["theta"]
    if kind == "neighbours":
        return None  # whole numbers
    reps = d["reps"]
    L, p0, v0 = (_per_cell(reps, f) for f in ("Lx", "p0", "v0"))
    amp = math.sqrt(2.0 * DR * DT)
    if kind == "eval":
        x, y = x.requires_grad_(True), y.requires_grad_(True)
        A, P, E = _spv_energy(x, y, L, _rings(x, y, reps), p0)
        gx, gy = torch.autograd.grad(E, (x, y))
        return None, None, A.detach(), P.detach(), -gx, -gy, float(E)
    if kind == "grad":
        leaf = [x, y, d["p0"]] + [torch.tensor(v, dtype=F64, device=DEV) for v in (case["v0"], 1.0, 1.0)]
        leaf = [t.requires_grad_(True) for t in leaf]
        x, y, p0, v0, KA, KP = leaf
        for k in range(case["steps"]):
            x, y = _spv_step(x, y, theta, reps, L, p0, v0, KA, KP, grad=True)
            theta = theta + amp * _noise(len(x), k, seed)
        A, P = _spv_geometry(x, y, L, _rings(x, y, reps))
        loss = _loss(A, P)
        loss.backward()
        return [t.detach() for t in (x, y, A, P, loss)] + [t.grad for t in leaf]
    xs, ys = [], []
    for k in range(case["steps"]):
        x, y = _spv_step(x, y, theta, reps, L, p0, d["v0"][k] if kind == "io" else v0)
        theta = theta + amp * _noise(len(x), k, seed, case.get("precision", "f64"))
        xs.append(x)
        ys.append(y)
    if kind == "io":
        return torch.stack([torch.stack(xs), torch.stack(ys)])
    return x, y, theta


# ---- vertex model --------------------------------------------------------
def _network(x, y, L):
    """The Voronoi network of seeds: vertices numbered by the triangles of
    each cell that is its smallest, in ring order from the smallest neighbour."""
    ring = _delaunay(x, y, L)
    n = len(x)
    cnt = (ring >= 0).sum(1)
    shift = torch.where(ring >= 0, ring, n).argmin(1)
    a = torch.arange(RING, device=ring.device).expand_as(ring)
    ring = torch.where(a < cnt[:, None], ring.gather(1, (a + shift[:, None]) % cnt[:, None]), -1)
    nx = _next(ring, cnt)
    i = torch.arange(n, device=ring.device)[:, None].expand_as(ring)
    tri = torch.stack([i, ring, ring.gather(1, nx)], -1)
    used = ring >= 0
    s = tri.sort(-1).values
    key = torch.where(used, (s[..., 0] * n + s[..., 1]) * n + s[..., 2], -1)
    own = used & (i < tri[..., 1]) & (i < tri[..., 2])
    okey, back = key[own].sort()
    cv = torch.where(used, back[torch.searchsorted(okey, key.clamp(min=0)).clamp(max=len(okey) - 1)], -1)
    vc = tri[own]
    o = vc[:, 0]

    def before(c, v):  # the vertex before v in cell c's list
        at = (cv[c] == v[:, None]).long().argmax(1)
        return cv[c, (at - 1) % cnt[c]]

    v = torch.arange(len(vc), device=x.device)
    vn = torch.stack([before(c, v) for c in (vc[:, 0], vc[:, 1], vc[:, 2])], 1)
    j, k = vc[:, 1], vc[:, 2]
    ax, ay, bx, by = (_image(q[t] - q[o], L) for t in (j, k) for q in (x, y))
    det = 2.0 * (ax * by - ay * bx)
    la, lb = ax * ax + ay * ay, bx * bx + by * by
    hx, hy = x[o] + (by * la - ay * lb) / det, y[o] + (ax * lb - bx * la) / det
    return torch.remainder(hx, L), torch.remainder(hy, L), vc, vn, cnt, cv


def _t1_passes(hx, hy, vc, vn, cc, cv, L):
    """T1 passes on numpy arrays, in place: short edges whose id (3 times the
    smaller end plus its slot) is the smallest on all four of their cells
    rotate by 90 degrees; repeated until none is short."""
    img = lambda q: q - L * np.round(q / L)  # noqa: E731
    for _ in range(16):
        V = len(hx)
        w = vn.reshape(-1)
        v = np.repeat(np.arange(V), 3)
        l2 = img(hx[w] - hx[v]) ** 2 + img(hy[w] - hy[v]) ** 2
        ids = np.nonzero((v < w) & (l2 < T1_THRESHOLD ** 2))[0]
        cand, best = [], {}
        for e in ids:
            v1, a = divmod(int(e), 3)
            v2 = int(vn[v1, a])
            i, k, j = (int(vc[v1, (a + q) % 3]) for q in range(3))
            l = next(int(c) for c in vc[v2] if c not in (i, k))
            if cc[i] > 3 and cc[k] > 3 and cc[j] < RING and cc[l] < RING:
                cand.append((int(e), v1, a, v2, i, j, k, l))
                for c in (i, j, k, l):
                    best[c] = min(best.get(c, 1 << 62), int(e))
        if not cand:
            return
        for e, v1, a, v2, i, j, k, l in cand:
            if any(best[c] != e for c in (i, j, k, l)):
                continue
            b = list(vn[v2]).index(v1)
            up, low = vn[v1, (a + 1) % 3], vn[v1, (a + 2) % 3]  # v1's outer neighbours
            lr, ur = vn[v2, (b + 1) % 3], vn[v2, (b + 2) % 3]   # v2's
            ex, ey = img(hx[v2] - hx[v1]), img(hy[v2] - hy[v1])
            mx, my = hx[v1] + 0.5 * ex, hy[v1] + 0.5 * ey
            h = 0.75 * T1_THRESHOLD / math.hypot(ex, ey)
            hx[v1], hy[v1] = (mx + ey * h) % L, (my - ex * h) % L
            hx[v2], hy[v2] = (mx - ey * h) % L, (my + ex * h) % L
            vc[v1], vn[v1] = (j, i, l), (low, lr, v2)
            vc[v2], vn[v2] = (k, j, l), (up, v1, ur)
            vn[up][list(vn[up]).index(v1)] = v2
            vn[lr][list(vn[lr]).index(v2)] = v1
            rows = {c: list(cv[c, :cc[c]]) for c in (i, j, k, l)}
            rows[i].remove(v2)
            rows[k].remove(v1)
            rows[j].insert(rows[j].index(v1) + 1, v2)
            rows[l].insert(rows[l].index(v2) + 1, v1)
            for c, row in rows.items():
                cc[c] = len(row)
                cv[c] = row + [-1] * (RING - len(row))


def _exact_avm(case, seed, d):
    L, theta = d["L"], d["theta"]
    hx, hy, vc, vn, cc, cv = _network(d["x"], d["y"], L)
    amp = math.sqrt(2.0 * DR * DT)
    for k in range(case["steps"]):
        x, y = hx.detach().requires_grad_(True), hy.detach().requires_grad_(True)
        used = cv >= 0
        row = torch.where(used, cv, cv[:, :1])
        px, py = _image(x[row] - x[row[:, :1]], L), _image(y[row] - y[row[:, :1]], L)
        nx = _next(cv, cc)
        qx, qy = px.gather(1, nx), py.gather(1, nx)
        A = 0.5 * torch.where(used, px * qy - qx * py, 0.0).sum(1)
        P = torch.where(used, torch.sqrt(torch.where(used, (qx - px) ** 2 + (qy - py) ** 2, 1.0)), 0.0).sum(1)
        gx, gy = torch.autograd.grad(((A - 1.0) ** 2 + (P - 3.8) ** 2).sum(), (x, y))
        ax, ay = (0.1 / 3.0 * f(theta)[vc].sum(1) for f in (torch.cos, torch.sin))
        hx, hy = torch.remainder(hx + DT * (ax - gx), L), torch.remainder(hy + DT * (ay - gy), L)
        net = [t.cpu().numpy() for t in (hx, hy, vc, vn, cc, cv)]
        _t1_passes(*net, L)
        hx, hy, vc, vn, cc, cv = (torch.from_numpy(t).to(DEV) for t in net)
        theta = theta + amp * _noise(case["n"], k, seed)
    return [hx, hy, theta, None, None, None, None]
