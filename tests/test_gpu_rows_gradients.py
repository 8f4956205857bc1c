"""The row sorts of a graph's construction at the lengths where the sort used
changes, and the policy's gradient at batch sizes around a warp's and the
grid's share of samples."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from oracle import mlp as omlp

sp = pytest.importorskip("paper_1903_12085_gb300")
torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    yield
    sp.set_tuning()


@pytest.mark.parametrize("top", [9, 1 << 24])
@pytest.mark.parametrize("degrees", [
    [2, 31, 32, 33, 63, 64, 65, 127, 128, 129],
    [4095, 4096, 4097, 8191, 8192, 8193, 12289, 128, 33],
    [16385, 70000, 4097, 24576] + [5000] * 40,
], ids=["warp", "chunks", "merges"])
def test_rows_of_every_length(degrees, top):
    """Rows of each length, out of order and with equal costs; IN-SIMPLE and
    OUT-SIMPLE take a row's first unsettled edge, so a row out of order shows
    in the settled sets."""
    rng = np.random.default_rng(len(degrees) + top)
    k, n = len(degrees), 6000
    u = np.concatenate([np.repeat(np.arange(k), degrees), np.arange(n)])
    v = np.concatenate([rng.integers(0, n, sum(degrees)), (np.arange(n) * 7 + 1) % n])
    w = rng.integers(0, top, len(u))
    for a, b in ((u, v), (v, u)):  # long rows, long in-rows
        g = gg.from_edges(n, list(zip(a.tolist(), b.tolist(), w.tolist())))
        G = sp.Graph.from_csr(g, reverse=True)
        ref = oracle.dijkstra(g, 0)
        for crit in (sp.IN_OUT, sp.SIMPLE):
            sim = oracle.simulate(g, 0, crit, dist_ref=ref)
            dist, st, settle, _ = sp.solve_trace(G, 0, crit, trace_cap=1 << 16)
            assert (sp.as_uint64(dist) == ref).all()
            assert st["phases"] == sim.phases and (settle == sim.settle_phase).all()
        G.close()


@pytest.mark.parametrize("batch", [1, 2, 7, 8, 9, 1215, 1217, 9727, 9729, 30001])
def test_gradient_batch_sizes(batch):
    """Against float64.  A gradient is a sum of `batch` FP32 terms of which a
    lane adds at most batch / 1216 + 8 in a row: 1e-4 of the largest entry is
    what the fixed batch of the other gradient test is held to as well."""
    rng = np.random.default_rng(batch)
    w = omlp.init(11).astype(np.float32)
    x = rng.uniform(0, 1, size=(batch, 8)).astype(np.float32)
    t = rng.normal(0, 2, size=batch).astype(np.float32)
    a = rng.integers(0, 4, size=batch).astype(np.uint32)
    cu = [torch.from_numpy(v.view(np.int32) if v.dtype == np.uint32 else v).cuda() for v in (w, x, t, a)]
    g, loss = sp.mlp_backward(*cu)
    L, ref = omlp.backward(w.astype(np.float64), x.astype(np.float64), t.astype(np.float64), a)
    assert np.isclose(float(loss.item()), L, rtol=1e-4)
    assert np.abs(g.cpu().numpy() - ref).max() <= 1e-4 * np.abs(ref).max()
    assert torch.equal(g, sp.mlp_backward(*cu)[0])
