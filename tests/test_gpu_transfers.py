"""Getters and setters with the caller's buffers on the device (read and written
in place), in host memory and on the device without the alignment of a vector
store (both staged): the same values."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1702_02939_gb300 as cg
import workloads

pytestmark = pytest.mark.gpu


def _buffers(where, n, dtype):
    if where == "host":
        return np.zeros(n, np.float64 if dtype == torch.float64 else np.int32)
    pad = 1 if where == "offset" else 0  # one element past an aligned start
    return torch.zeros(n + pad, dtype=dtype, device="cuda")[pad:]


def _np(b):
    return b if isinstance(b, np.ndarray) else b.cpu().numpy()


@pytest.mark.parametrize("n", [97, 4099])
def test_spv_transfers(n):
    x, y, th, L = workloads.spv_uniform(n, 4)
    sim = cg.SPV([dict(n=n, Lx=L, Ly=L, p0=3.8, v0=0.1)], x, y, th, dt=0.005, seed=2)
    sim.step(3)
    got = {}
    for where in ("device", "host", "offset"):
        d = [_buffers(where, n, torch.float64) for _ in range(7)]
        cnt, nbr = _buffers(where, n, torch.int32), _buffers(where, 16 * n, torch.int32)
        cg.cg_get_state(sim.ctx, *d[:3])
        cg.cg_get_geometry(sim.ctx, *d[3:5])
        E = cg.cg_get_forces(sim.ctx, *d[5:])
        cg.cg_get_neighbors(sim.ctx, cnt, nbr)
        got[where] = [_np(b) for b in (*d, cnt, nbr)] + [np.array(E)]
        cg.cg_set_state(sim.ctx, *d[:3])  # the same state back
        cg.cg_set_p0(sim.ctx, _buffers(where, n, torch.float64) + 3.8)
    for where in ("host", "offset"):
        for a, b in zip(got["device"], got[where]):
            assert np.array_equal(a, b)
    A, P = got["device"][3:5]
    assert float(got["device"][-1]) == pytest.approx(float(((A - 1) ** 2 + (P - 3.8) ** 2).sum()), rel=1e-13)
    sim.close()


@pytest.mark.parametrize("sort_every", [0, 2])
def test_vertex_model_transfers(sort_every):
    n = 301
    x, y, th, L = workloads.spv_uniform(n, 4)
    sim = cg.AVM(n, L, L, x, y, th, v0=0.3, seed=2, sort_every=sort_every)
    sim.step(5)
    got = {}
    for where in ("device", "host", "offset"):
        d = [_buffers(where, k, torch.float64) for k in (2 * n, 2 * n, n)]
        i = [_buffers(where, k, torch.int32) for k in (6 * n, 6 * n, n, 16 * n)]
        cg.cg_avm_get_state(sim.ctx, *d)
        cg.cg_avm_get_topology(sim.ctx, *i)
        got[where] = [_np(b) for b in (*d, *i)]
    for where in ("host", "offset"):
        for a, b in zip(got["device"], got[where]):
            assert np.array_equal(a, b)
    sim.close()


@pytest.mark.parametrize("sort_every", [0, 20])
def test_many_steps_per_launch_equal_single_steps(sort_every):
    """Past the first 64 steps a call's steps go several per graph launch; the
    result is that of one call per step, through re-sorts and changed moduli."""
    n = 150
    x, y, th, L = workloads.spv_uniform(n, 6)
    for make in (lambda: cg.SPV([dict(n=n, Lx=L, Ly=L, p0=3.8, v0=0.2)], x, y, th, seed=3, sort_every=sort_every),
                 lambda: cg.AVM(n, L, L, x, y, th, v0=0.2, seed=3, sort_every=sort_every)):
        got = []
        for single in (False, True):
            sim = make()
            for steps in (70, 19, 7, 33):
                for _ in range(steps if single else 1):
                    sim.step(1 if single else steps)
                if isinstance(sim, cg.SPV) and steps == 19:
                    sim.set_moduli(1.5, 0.5)
            got.append([t.cpu().numpy() for t in sim.state()])
            sim.close()
        for a, b in zip(*got):
            assert np.array_equal(a, b)
