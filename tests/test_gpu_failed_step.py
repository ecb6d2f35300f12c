"""A step that raises a status: the getters that follow return it and leave the
caller's buffers as they are."""
import pytest

torch = pytest.importorskip("torch")

import paper_1702_02939_gb300 as cg
import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sort_every", [0, 50])
def test_vertex_model_getters_after_a_failed_step(sort_every):
    n = 400
    x, y, th, L = workloads.spv_uniform(n, 3)
    # a fresh network needs more than one pass at this threshold
    mk = lambda: cg.AVM(n, L, L, x, y, th, t1_threshold=0.2, t1_cap=1, sort_every=sort_every)
    for get, sizes, dtype in ((cg.cg_avm_get_topology, (6 * n, 6 * n, n, 16 * n), torch.int32),
                              (cg.cg_avm_get_state, (2 * n, 2 * n, n), torch.float64)):
        sim = mk()
        out = [torch.full((k,), -7, dtype=dtype, device="cuda") for k in sizes]
        sim.step(1)  # the status is not read here
        with pytest.raises(cg.CellgbError):
            get(sim.ctx, *out)
        assert all(bool((b == -7).all()) for b in out)
        sim.close()
