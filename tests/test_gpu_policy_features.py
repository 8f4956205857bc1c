"""What the engine's warps see of a phase is what the host function computes
from the phase's record: the arms of a traced policy solve are those that the
forward kernel and the documented choice give on the host's features."""
import numpy as np
import pytest

import graphgen as gg
from oracle import mlp as omlp

sp = pytest.importorskip("paper_1903_12085_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

MARGIN = 0.35  # by which an arm has to beat arm 0


def test_arms_follow_from_the_host_features():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    got = [_follow(seed) for seed in range(4)]
    assert min(n for n, _ in got) > 50 and len(set().union(*(arms for _, arms in got))) > 1


def _follow(seed):
    """Checks one network; how many phases were not too close to call, and their arms."""
    w = omlp.init(500 + seed, scale=1.0).astype(np.float32)
    sp.policy_load(w)
    sp.set_tuning()
    sp.set_tuning(solo_max_frontier=0, nearfar_min_frontier=0)  # all blocks: asked in phases 1, 5, 9, ...
    checked, arms = 0, set()
    try:
        for g in (gg.gnm(4000, 30000, 0, 1 << 24, 81), gg.rmat(12, 12, 0.57, 0.19, 0.19, 0, 1 << 24, 82),
                  gg.grid(40, 50, 1, 1 << 16, 83)):
            G = sp.Graph.from_csr(g, reverse=True)
            _, _, _, tr = sp.solve_trace(G, 1, sp.IN_OUT | sp.POLICY_LEARNED, trace_cap=1 << 16)
            prev = np.zeros(1, tr.dtype)[0]
            asked = []
            for k, r in enumerate(tr, start=1):
                if k % 4 == 1:
                    asked.append((r, sp.policy_features(r["frontier"], G.n, G.m, k, prev["deg_settled"], prev["settled"],
                                                        prev["frontier"])))
                prev = r
            x = torch.from_numpy(np.array([f for _, f in asked], np.float32)).cuda()
            ys = sp.mlp_forward(torch.from_numpy(w).cuda(), x).cpu().numpy()
            for (r, _), y in zip(asked, ys):
                may = [a for a in range(4) if a % 2 == 0 or int(r["frontier"]) * 32 >= G.n]
                order = sorted(may, key=lambda a: y[a])
                gap = min(abs(y[order[0]] - (y[0] - MARGIN)), y[order[1]] - y[order[0]])
                if gap < 1e-4 * (1 + np.abs(y).max()):
                    continue  # (too close to call: the two forward passes add in different orders)
                want = order[0] if y[order[0]] < y[0] - MARGIN else 0
                assert (int(r["arm"]) >> 8) & 3 == want, (g.name, y, int(r["frontier"]))
                arms.add(want)
                checked += 1
    finally:
        sp.set_tuning()
        sp.policy_clear()
    return checked, arms
