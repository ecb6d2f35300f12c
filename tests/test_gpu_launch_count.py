"""The benchmark's count of its own launches against the profiler's, at every form
of the step graph."""
import pytest

torch = pytest.importorskip("torch")

import bench
import paper_1702_02939_gb300 as cg
import workloads

pytestmark = pytest.mark.gpu


def _launched(run):
    from torch.profiler import ProfilerActivity, profile

    with profile(activities=[ProfilerActivity.CUDA, ProfilerActivity.CPU]) as p:
        run()
        torch.cuda.synchronize()
    return sum("cgk::k_" in e.name for e in p.events())


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("n", [1000, 4000, 20000, 60000, 200000])
def test_kernels_of_a_step(n, precision):
    x, y, th, L = workloads.spv_uniform(n, 1)
    sim = cg.SPV([dict(n=n, Lx=L, Ly=L, p0=3.85, v0=0.1)], x, y, th, dt=0.001, seed=1, precision=precision)
    if not _launched(lambda: sim.step(1)) and not _launched(lambda: sim.step(1)):
        pytest.skip("the profiler sees no kernel")
    c0 = sim.counters()
    got = _launched(lambda: sim.step(5))
    c = sim.counters()
    assert got == bench.kernels_launched(5, c["loop_total"] - c0["loop_total"], n,
                                         ring_order=cg.cg_get_launch(sim.ctx)["ring_order"], fp32=precision == "f32")
    sim.close()
