"""Criteria whose phases on one block are the generic ones, with the fringe in
global memory: a large solo_max_frontier stands for 2048 vertices, and a fringe
beyond that is run by all blocks."""
import pytest

import graphgen as gg
import oracle

sp = pytest.importorskip("paper_1903_12085_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("limit,largest", [(1 << 31, 2048), (2048, 2048), (300, 300)])
@pytest.mark.parametrize("crit", [sp.SIMPLE, sp.IN_FULL | sp.OUT_WEAK], ids=["simple", "full_weak"])
def test_largest_fringe_on_one_block(crit, limit, largest):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = gg.gnm(20000, 160000, 0, 1 << 24, 91)
    ref = oracle.dijkstra(g, 0)
    G = sp.Graph.from_csr(g, reverse=True)
    try:
        sp.set_tuning()
        sp.set_tuning(solo_max_frontier=limit)
        dist, st, _, recs = sp.solve_trace(G, 0, crit, trace_cap=1 << 12)
    finally:
        sp.set_tuning()
    assert (sp.as_uint64(dist) == ref).all()
    assert st["phases"] == oracle.simulate(g, 0, crit, dist_ref=ref).phases
    one_block = (recs["arm"] & 2) != 0
    assert recs["frontier"].max() > 2048  # (both kinds of phases occur)
    assert (one_block == (recs["frontier"] <= largest)).all()
