"""A prepared batch keeps the tuning it was created with when records are
attached to it and taken off again (which changes its kernel instance)."""
import pytest

import graphgen as gg
import oracle

sp = pytest.importorskip("paper_1903_12085_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ON_ONE_BLOCK = 2  # bit of a record's arm word


@pytest.mark.parametrize("created,later", [(dict(solo_max_frontier=0), {}), ({}, dict(solo_max_frontier=0))],
                         ids=["no_episodes", "episodes"])
def test_tuning_of_creation_outlasts_a_trace(created, later):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = gg.gnm(3000, 24000, 0, 1 << 24, 81)
    ref = oracle.dijkstra(g, 2)
    phases = oracle.simulate(g, 2, sp.IN_OUT, dist_ref=ref).phases
    try:
        sp.set_tuning()
        sp.set_tuning(batch_blocks_per_solve=3, **created)
        b = sp.Batch([sp.Graph.from_csr(g)] * 2, [2, 2], sp.IN_OUT)
        sp.set_tuning()
        sp.set_tuning(**later)
        for _ in range(2):
            b.attach_trace(1, 1 << 12)
            b.launch()
            torch.cuda.synchronize()
            _, recs = b.trace_of(1)
            assert len(recs) == phases
            assert ((recs["arm"] & ON_ONE_BLOCK) != 0).any() == ("solo_max_frontier" not in created)
            b.detach_trace(1)
            for o in b.outs:
                o.zero_()
            b.launch()
            torch.cuda.synchronize()
            assert all((sp.as_uint64(o) == ref).all() for o in b.outs) and b.phases.tolist() == [phases] * 2
        b.close()
    finally:
        sp.set_tuning()
