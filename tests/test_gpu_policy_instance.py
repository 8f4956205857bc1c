"""Untraced policy solves run in an instance of their own, which keeps no status
bytes; traced ones in the general instance, whose schedules other tests replay
in the oracle.  Both choose from the same features, so distances and phase
counts must be the same, whatever arms a network picks.  (With a forced
near/far split only the distances: the bound follows the fills of the bucket
lists, which depend on the order of the relaxations, and while the fringe is
split a policy's choice rests, so the phases it is asked in vary from run to
run.)"""
import numpy as np
import pytest

import graphgen as gg
import oracle
from oracle import mlp as omlp

sp = pytest.importorskip("paper_1903_12085_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

LEARNED = sp.IN_OUT | sp.POLICY_LEARNED
TUNINGS = {"default": {}, "one_block": dict(grid_blocks=1), "no_episodes": dict(solo_max_frontier=0),
           "short_episodes": dict(grid_blocks=3, solo_max_edges=24, solo_max_frontier=90),
           "split": dict(grid_blocks=3, nearfar_min_frontier=8, nearfar_target=40, nearfar_min_share=0)}


@pytest.fixture(params=list(TUNINGS))
def tuning(request):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sp.set_tuning()
    sp.set_tuning(**TUNINGS[request.param])
    yield request.param
    sp.set_tuning()
    sp.policy_clear()


def always(arm):
    """A network that prefers one arm by more than the margin."""
    w = np.zeros(sp.POLICY_WEIGHTS, np.float32)
    w[-4:] = 2.0
    w[-4 + arm] = 0.0
    return w


@pytest.mark.parametrize("net", ["arm0", "arm1", "arm2", "arm3", "mixed5", "mixed6"])
def test_untraced_and_traced_policy_solves_agree(net, tuning):
    sp.policy_load(always(int(net[3])) if net[:3] == "arm" else omlp.init(300 + int(net[5:]), scale=1.0).astype(np.float32))
    fixed = tuning != "split"
    for g in (gg.gnm(3000, 20001, 0, 1 << 24, 71), gg.rmat(11, 9, 0.57, 0.19, 0.19, 0, 1 << 24, 72),
              gg.grid(40, 77, 1, 1 << 16, 73), gg.gnm(70, 200, 0, 5, 74)):
        G = sp.Graph.from_csr(g, reverse=True)
        src = [1, g.n // 2, g.n - 1]
        refs = [oracle.dijkstra(g, s) for s in src]
        for s, ref in zip(src, refs):
            dist, st, _, tr = sp.solve_trace(G, s, LEARNED, trace_cap=1 << 16)
            assert (sp.as_uint64(dist) == ref).all()
            dist, phases = sp.solve(G, s, LEARNED)
            assert (sp.as_uint64(dist) == ref).all() and (phases == st["phases"] or not fixed), (g.name, s)
        if tuning in ("default", "split") and g.n > 100:
            for copies in (2, 110):  # blocks of 512 threads, and more solves than SMs of one size
                outs, phases = sp.solve_batch([G] * (3 * copies), src * copies, LEARNED)
                assert all((sp.as_uint64(o) == refs[i % 3]).all() for i, o in enumerate(outs)), g.name
                assert not fixed or len(set(phases[0::3])) == len(set(phases[1::3])) == len(set(phases[2::3])) == 1, g.name
        G.close()
