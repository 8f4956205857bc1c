"""Episodes on one block of a group: the group's blocks and the leading block
take the same decision in every phase, whatever way an episode ends.  Each
solve has many short episodes (hand-offs, overflows, pulls and the generic
phases of the dynamic criteria); a missing or surplus arrival would end it in a
timeout, another decision in other settled sets."""
import pytest

import graphgen as gg
import oracle

sp = pytest.importorskip("paper_1903_12085_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ENDS = {"hand_offs": dict(solo_max_edges=24), "overflows": dict(solo_max_frontier=60), "default": {},
        "pulls": dict(nearfar_min_frontier=8, nearfar_target=40, nearfar_min_share=0)}


@pytest.fixture(params=list(ENDS))
def ends(request):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sp.set_tuning()
    sp.set_wait_limit_ns(2_000_000_000)
    yield ENDS[request.param]
    sp.set_tuning()


@pytest.mark.parametrize("crit", [sp.IN_OUT, sp.IN_SIMPLE | sp.OUT_STATIC, sp.SIMPLE, sp.IN_FULL | sp.OUT_WEAK])
def test_groups_and_their_leader_agree(crit, ends):
    for g in (gg.gnm(2500, 20000, 0, 1 << 24, 61), gg.rmat(11, 15, 0.57, 0.19, 0.19, 0, 1 << 24, 62),
              gg.grid(45, 47, 1, 1 << 16, 63)):
        G = sp.Graph.from_csr(g, reverse=True)
        ref = oracle.dijkstra(g, 1)
        sim = oracle.simulate(g, 1, crit, dist_ref=ref)
        for blocks in (2, 7, 1 << 16):  # (1 << 16: every co-resident block)
            sp.set_tuning(grid_blocks=blocks, batch_blocks_per_solve=min(blocks, 16), **ends)
            for _ in range(5):
                dist, st, settle, _ = sp.solve_trace(G, 1, crit)
                assert (sp.as_uint64(dist) == ref).all() and (settle == sim.settle_phase).all(), (g.name, blocks)
                dist, phases = sp.solve(G, 1, crit)
                assert (sp.as_uint64(dist) == ref).all() and phases == sim.phases, (g.name, blocks)
            outs, phases = sp.solve_batch([G] * 12, [1] * 12, crit)
            assert all((sp.as_uint64(o) == ref).all() for o in outs) and (phases == sim.phases).all(), (g.name, blocks)
        G.close()


@pytest.mark.parametrize("edges", [0, 1, 7, 2048, 0xFFFFFFFF])
def test_edge_limits_of_an_episode(edges):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    try:
        for g in (gg.rmat(11, 19, 0.57, 0.19, 0.19, 0, 1 << 24, 64), gg.gnm(900, 30000, 0, 1 << 24, 65)):
            G = sp.Graph.from_csr(g)
            ref = oracle.dijkstra(g, 1)
            sim = oracle.simulate(g, 1, sp.IN_OUT, dist_ref=ref)
            for blocks in (1, 3):
                sp.set_tuning()
                sp.set_tuning(solo_max_edges=edges, grid_blocks=blocks)
                dist, st, settle, _ = sp.solve_trace(G, 1, sp.IN_OUT)
                assert (sp.as_uint64(dist) == ref).all() and (settle == sim.settle_phase).all(), (g.name, blocks)
                assert (st["settled"], st["edges_relaxed"]) == (sim.settled, sim.relaxed)
                dist, phases = sp.solve(G, 1, sp.IN_OUT)
                assert (sp.as_uint64(dist) == ref).all() and phases == sim.phases, (g.name, blocks)
    finally:
        sp.set_tuning()
