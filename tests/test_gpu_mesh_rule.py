"""Which graphs get a mesh's layout and launch plan hangs on their longest row:
rows on both sides of the limit, sizes on both sides of the one from which it
counts, alone and mixed in a batch, against the oracle."""
import numpy as np
import pytest

import graphgen as gg
import oracle

sp = pytest.importorskip("paper_1903_12085_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def ring(n, degree, wmax, seed):
    """Vertex i to i+1 .. i+degree, all rows of one length."""
    rng = np.random.default_rng(seed)
    u = np.repeat(np.arange(n), degree)
    v = (u + 1 + np.tile(np.arange(degree), n)) % n
    w = rng.integers(0, wmax, len(u))
    return gg.from_edges(n, list(zip(u.tolist(), v.tolist(), w.tolist())), f"ring{degree}")


@pytest.fixture(autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sp.set_tuning()


@pytest.mark.parametrize("degree", [1, 8, 9])
@pytest.mark.parametrize("n", [1 << 17, (1 << 17) + 1])
def test_single_solves(n, degree):
    if degree == 1 and n > 1 << 17:
        n = 3000  # (a chain: a phase per vertex)
    elif degree == 1:
        n = 1
    g = ring(n, degree, 1 << 20, degree) if n > 1 else gg.from_edges(1, [], "vertex")
    G = sp.Graph.from_csr(g)
    ref = oracle.dijkstra(g, 0)
    dist, phases = sp.solve(G, 0, sp.IN_OUT)
    assert (sp.as_uint64(dist) == ref).all() and 0 < phases <= g.n


@pytest.mark.parametrize("crit", [sp.IN_OUT, sp.IN_SIMPLE | sp.OUT_STATIC])
def test_mixed_batches(crit):
    """Sparse graphs that are no meshes (stages of several blocks, few slots in
    small blocks), meshes, and a large mesh beside a graph that is none."""
    rng = np.random.default_rng(9)
    sparse = [gg.gnm(n, int(4.5 * n), 0, 1 << 20, n) for n in (60000, 9000, 900, 700)]
    even = [gg.gnm(1200, 5000, 0, 1 << 20, 61 + i) for i in range(3)]
    large_mesh, beside = gg.grid(366, 360, 1, 1 << 16, 62), gg.gnm(1 << 17, 1 << 19, 0, 1 << 20, 63)
    for graphs, reps in ((sparse, 50), (even, 110), ([ring(800, 8, 1 << 20, 1), gg.grid(28, 29, 1, 99, 2)], 160),
                         ([large_mesh, beside] + even, 2)):
        pick = [g for g in graphs for _ in range(1 if g.n > 50000 else reps)]
        src = [int(rng.integers(g.n)) for g in pick]
        handles = {id(g): sp.Graph.from_csr(g, reverse=True) for g in graphs}
        outs, phases = sp.solve_batch([handles[id(g)] for g in pick], src, crit)
        for i, (g, s, o, ph) in enumerate(zip(pick, src, outs, phases)):
            ref = oracle.dijkstra(g, s)
            assert (sp.as_uint64(o) == ref).all(), g.name
            if g.n < 5000 and i % 8 == 0:
                assert ph == oracle.simulate(g, s, crit, dist_ref=ref).phases, g.name
