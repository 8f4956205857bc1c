"""Batches of more solves than SMs and of one size run in blocks of 256 threads,
with shared-memory layouts of their own: 32- and 64-bit distances, with few and
with many slots, the policy's weights behind them, and a split fringe.  Each
against the oracle."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from oracle import mlp as omlp

sp = pytest.importorskip("paper_1903_12085_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

NARROW = 1 << 29  # largest cost that the 32-bit slots take
SPLIT = dict(nearfar_min_frontier=8, nearfar_target=40, nearfar_min_share=0)
FAMILIES = {"mesh": lambda lo, hi, seed: gg.grid(33, 47, lo, hi, seed),  # many slots a thread
            "dense": lambda lo, hi, seed: gg.gnm(1500, 15003, lo, hi, seed)}  # few


@pytest.fixture(params=[{}, SPLIT], ids=["default", "split"])
def tuning(request):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sp.set_tuning()
    sp.set_tuning(**request.param)
    yield request.param
    sp.set_tuning()
    sp.policy_clear()


def solve(graphs, crit, solves=320):
    """`solves` solves of one size, more than any GPU of this kind has SMs."""
    src = [(7 * i) % graphs[0].n for i in range(solves)]
    handles = [sp.Graph.from_csr(g, reverse=True) for g in graphs]
    pick = [i % len(graphs) for i in range(solves)]
    outs, phases = sp.solve_batch([handles[p] for p in pick], src, crit)
    refs = [oracle.dijkstra(graphs[p], s) for p, s in zip(pick, src)]
    for o, ref in zip(outs, refs):
        assert (sp.as_uint64(o) == ref).all()
    return [(graphs[p], s, ref, int(ph)) for p, s, ref, ph in zip(pick, src, refs, phases)]


@pytest.mark.parametrize("family", list(FAMILIES))
@pytest.mark.parametrize("wmax", [100, NARROW, NARROW + 1, 0xFFFFFFFE])
def test_widths_and_slots(wmax, family, tuning):
    graphs = [FAMILIES[family](lo, wmax + 1, 101 + i) for i, lo in enumerate((0, wmax - 5))]
    for crit in (sp.IN_OUT, sp.IN_SIMPLE | sp.OUT_STATIC):
        for g, s, ref, phases in solve(graphs, crit)[::16]:
            assert phases == oracle.simulate(g, s, crit, dist_ref=ref).phases


@pytest.mark.parametrize("family", list(FAMILIES))
@pytest.mark.parametrize("wmax", [1 << 20, NARROW + 1])
def test_policy(wmax, family, tuning):
    sp.policy_load(omlp.init(401, scale=1.0).astype(np.float32))
    graphs = [FAMILIES[family](1, wmax + 1, 111)]
    got = solve(graphs, sp.IN_OUT | sp.POLICY_LEARNED)
    if tuning:
        return  # (the phases a policy is asked in then vary from run to run)
    G = sp.Graph.from_csr(graphs[0], reverse=True)
    sp.set_tuning(grid_blocks=1)
    for g, s, ref, phases in got[::16]:
        assert phases == sp.solve_trace(G, s, sp.IN_OUT | sp.POLICY_LEARNED)[1]["phases"]
