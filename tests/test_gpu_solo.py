"""Solo episodes (fringe in shared memory) and the kernels' plain instances
against the oracle: costs on both sides of the 32-bit limit, distances that run
far past 2^32, rows longer than a warp or a phase takes, fringes that outgrow
the slots, and the switch between the instances when a batch records."""
import numpy as np
import pytest

import graphgen as gg
import oracle

sp = pytest.importorskip("paper_1903_12085_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

NARROW = 1 << 29  # largest cost that the 32-bit slots take
TUNINGS = {"default": {}, "one_block": dict(grid_blocks=1), "few_edges_3blk": dict(grid_blocks=3, solo_max_edges=24),
           "cap_100": dict(solo_max_frontier=100),
           "split_small": dict(grid_blocks=3, nearfar_min_frontier=8, nearfar_target=40, nearfar_min_share=0)}


@pytest.fixture(params=list(TUNINGS))
def tuning(request):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sp.set_tuning()
    sp.set_tuning(**TUNINGS[request.param])
    yield request.param
    sp.set_tuning()


def race(n, heavy):
    """A chain of `heavy` edges beside a chain of unit ones, crossed now and then:
    with IN-SIMPLE the heavy chain runs away from the light one."""
    edges = [(0, 1, heavy), (0, n, 1)]
    edges += [(i, i + 1, heavy) for i in range(1, n - 1)] + [(n + i, n + i + 1, 1) for i in range(n - 1)]
    edges += [(i, n + i + 1, heavy) for i in range(0, n - 1, 7)]
    return gg.from_edges(2 * n, edges, f"race{n}")


def graphs(wmax):
    lo = wmax - 5
    hub = [(0, v, 1 + v % 97) for v in range(1, 70001)] + [(v, 0, 3) for v in range(1, 50)]
    return [gg.gnm(3000, 24000, 0, wmax + 1, 11), gg.gnm(40, 60, lo, wmax + 1, 12), gg.grid(37, 91, lo, wmax + 1, 13),
            gg.rmat(11, 16, 0.57, 0.19, 0.19, 0, wmax + 1, 14), race(90, wmax),
            gg.from_edges(70001, hub + [(0, 1, wmax)], "hub")]


@pytest.mark.parametrize("wmax", [100, NARROW, NARROW + 1, 0xFFFFFFFE])
def test_costs_and_rows(wmax, tuning):
    for g in graphs(wmax):
        G = sp.Graph.from_csr(g, reverse=True)
        ref = oracle.dijkstra(g, 0)
        for crit in (sp.IN_OUT, sp.IN_STATIC, sp.OUT_STATIC, sp.IN_SIMPLE | sp.OUT_STATIC):
            if crit == sp.OUT_STATIC and "hub" in g.name:
                continue  # 70,000 phases or so
            sim = oracle.simulate(g, 0, crit, dist_ref=ref)
            dist, phases = sp.solve(G, 0, crit)  # static criteria: the plain instance, if the costs are narrow
            assert (sp.as_uint64(dist) == ref).all(), (g.name, crit)
            assert phases == sim.phases, (g.name, crit)
            dist, st, settle, _ = sp.solve_trace(G, 0, crit)
            assert (sp.as_uint64(dist) == ref).all() and (settle == sim.settle_phase).all(), (g.name, crit)
            assert (st["phases"], st["sum_frontier"], st["settled"], st["edges_relaxed"]) == \
                (sim.phases, sim.sum_f, sim.settled, sim.relaxed), (g.name, crit)
        G.close()


@pytest.mark.parametrize("n", [1 << 13, 1 << 16, (1 << 17) + 1])
def test_fringe_outgrows_the_slots(n, tuning):
    """A fringe that passes every limit on the way up and again on the way down."""
    g = gg.gnm(n, 5 * n + 7, 0, 1 << 24, 21)
    G = sp.Graph.from_csr(g)
    ref = oracle.dijkstra(g, 3)
    sim = oracle.simulate(g, 3, sp.IN_OUT, dist_ref=ref)
    dist, phases = sp.solve(G, 3, sp.IN_OUT)
    assert (sp.as_uint64(dist) == ref).all() and phases == sim.phases


def test_batch_of_both_widths_records_and_stops(tuning):
    gs = [gg.gnm(2000, 9000, 0, w, 31 + i) for i, w in enumerate([1 << 24, NARROW + 1])] + [gg.grid(40, 41, 1, 99, 33)]
    for pick in (gs, gs[:1] + gs[2:]):  # mixed (general instance), all narrow (plain until something records)
        G = [sp.Graph.from_csr(g) for g in pick]
        sims = [oracle.simulate(g, 5, sp.IN_OUT, dist_ref=oracle.dijkstra(g, 5)) for g in pick]
        b = sp.Batch(G, [5] * len(G), sp.IN_OUT)
        for step in ("plain", "traced", "plain again"):
            if step == "traced":
                b.attach_trace(0, 1 << 12)
            elif step == "plain again":
                b.detach_trace(0)
            for o in b.outs:
                o.zero_()
            b.launch()
            torch.cuda.synchronize()
            assert b.phases.tolist() == [s.phases for s in sims], step
            for g, o in zip(pick, b.outs):
                assert (sp.as_uint64(o) == oracle.dijkstra(g, 5)).all(), step
            if step == "traced":
                settle, recs = b.trace_of(0)
                assert (settle == sims[0].settle_phase).all() and len(recs) == sims[0].phases
        b.close()


@pytest.mark.parametrize("crit", [sp.IN_OUT, sp.IN_SIMPLE | sp.OUT_STATIC])
def test_batch_plans(crit):
    """One size and more solves than SMs (small blocks), uneven sizes (stages of
    several blocks per solve before the rest), meshes, and a single large solve
    among many small ones."""
    sp.set_tuning()
    rng = np.random.default_rng(5)
    even = [gg.gnm(400, 2500, 0, 1 << 20, 41 + i) for i in range(4)]
    uneven = [gg.gnm(n, 9 * n, 0, 1 << 20, n) for n in (40000, 9000, 3000, 700, 60)]
    mesh = [gg.grid(30, 31, 1, 1 << 16, 51), gg.grid(9, 200, 1, 1 << 16, 52)]
    for graphs, reps in ((even, 60), (uneven, 40), (mesh, 90), (uneven[:1] + even, 1), (mesh[:1] + uneven[1:2], 3)):
        pick = [g for g in graphs for _ in range(reps if g is not uneven[0] else min(reps, 3))]
        src = [int(rng.integers(g.n)) for g in pick]
        handles = {id(g): sp.Graph.from_csr(g, reverse=True) for g in graphs}
        outs, phases = sp.solve_batch([handles[id(g)] for g in pick], src, crit)
        for g, s, o, ph in zip(pick, src, outs, phases):
            ref = oracle.dijkstra(g, s)
            assert (sp.as_uint64(o) == ref).all()
            assert ph == oracle.simulate(g, s, crit, dist_ref=ref).phases
