"""The work that users of this library have it do, as timed cases.

Every case goes through the package's public calls on seeded graphs of the
families that the repository's workloads and tests are made of: uniform G(n, m)
(n from a thousand to 2^24 vertices, average degree 4 to 32), 4-neighbour grids
(deep: thousands of phases) and R-MAT graphs (power-law rows).  ``listed()``
names the cases, ``draw(rng)`` gives more of the same ranges with odd sizes.

The calls:
  solve   one single-source solve on a graph in hand (distances on the device)
  batch   several sources on one graph as a prepared batch, launched once
  uneven  several sources on each of many graphs of different sizes, one launch
  create  a one-off query from pinned host CSR: graph creation, solve,
          distances back in host memory
  train   one training step of the phase policy network (gradients and Adam)
"""
import math

import numpy as np
import torch

import paper_1903_12085_gb300 as sp

CRITERIA = {
    "in_out": sp.IN_OUT,
    "simple": sp.SIMPLE,
    "full_weak": sp.IN_FULL | sp.OUT_WEAK,
    "learned": sp.IN_OUT | sp.POLICY_LEARNED,
}
W24, W20, W16 = 1 << 24, 1 << 20, 1 << 16


def listed():
    return [
        # the smallest calls: a graph of a thousand vertices, where launch and phase latency are all
        {"name": "solve_gnm_1k", "call": "solve", "graph": "gnm", "n": 1000, "m": 8000, "wmax": W24,
         "criterion": "in_out"},
        # the ordinary single query of the study's uniform family
        {"name": "solve_gnm_16k", "call": "solve", "graph": "gnm", "n": 16384, "m": 131072, "wmax": W24,
         "criterion": "in_out"},
        # a road-like graph: 34 thousand dependent phases with a small fringe
        {"name": "solve_grid_1024", "call": "solve", "graph": "grid", "rows": 1024, "cols": 1024, "wmax": W16,
         "criterion": "in_out"},
        # a power-law graph with hub rows of tens of thousands of edges
        {"name": "solve_rmat_s22", "call": "solve", "graph": "rmat", "n": 1 << 22, "m": 1 << 26, "wmax": W24,
         "criterion": "in_out"},
        # the dynamic criteria (cursors over the reverse rows too) on a power-law graph
        {"name": "simple_rmat_s20", "call": "solve", "graph": "rmat", "n": 1 << 20, "m": 1 << 24, "wmax": W24,
         "criterion": "simple"},
        # the strongest criteria: fewest phases, most work in each; odd size
        {"name": "full_weak_gnm_300k", "call": "solve", "graph": "gnm", "n": 300007, "m": 3000071, "wmax": W24,
         "criterion": "full_weak"},
        # the largest single query
        {"name": "solve_gnm_16m", "call": "solve", "graph": "gnm", "n": 1 << 24, "m": 1 << 28, "wmax": W24,
         "criterion": "in_out"},
        # the largest step: 8 sources at once on the same graph, phases picked by a policy network
        {"name": "batch8_gnm_16m", "call": "batch", "graph": "gnm", "n": 1 << 24, "m": 1 << 28, "wmax": W24,
         "criterion": "learned", "sources": 8},
        # serving many queries on one road-like graph
        {"name": "batch256_grid_512", "call": "batch", "graph": "grid", "rows": 512, "cols": 512, "wmax": W16,
         "criterion": "in_out", "sources": 256},
        # many graphs of uneven size, 4 sources each, in one launch
        {"name": "uneven_256x4", "call": "uneven", "graphs": 256, "nmin": 1 << 10, "nmax": 1 << 18, "wmax": W20,
         "criterion": "in_out", "sources": 4},
        # a one-off query on a graph that has to be copied and prepared first
        {"name": "create_rmat_s20", "call": "create", "graph": "rmat", "n": 1 << 20, "m": 1 << 24, "wmax": W24,
         "criterion": "in_out"},
        # fitting the phase policy on the phases of its training solves
        {"name": "train_60k", "call": "train", "batch": 60000},
    ]


def _log_int(rng, lo, hi):
    """Integer in [lo, hi], uniform over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    call = rng.choice(["solve", "solve", "solve", "solve", "batch", "uneven", "create", "train"])
    if call == "train":
        return {"call": call, "batch": _log_int(rng, 1000, 60000)}
    if call == "uneven":
        return {"call": call, "graphs": _log_int(rng, 16, 256), "nmin": 1 << 10, "nmax": _log_int(rng, 1 << 13, 1 << 18),
                "wmax": W20, "criterion": "in_out", "sources": rng.randint(1, 4)}
    kind = rng.choice(["gnm", "grid", "rmat"])
    case = {"call": call, "graph": kind, "wmax": W16 if kind == "grid" else W24}
    if call == "batch":
        case["criterion"] = "in_out" if kind == "grid" else rng.choice(["in_out", "learned"])
        case["sources"] = _log_int(rng, 2, 256)
        # vertices of all the solves together: at most those of the listed batches
        top = ((1 << 26) if kind == "grid" else (1 << 27)) // case["sources"]
    elif call == "create":
        case["criterion"] = "in_out"
        top = 1 << 20
    else:
        case["criterion"] = "in_out" if kind == "grid" else rng.choice(["in_out", "in_out", "simple", "full_weak"])
        top = 1 << 24 if case["criterion"] == "in_out" else 1 << 20 if kind == "rmat" else 300007
    if kind == "grid":
        side = 1024 if call == "solve" else min(512, math.isqrt(top))
        case["rows"], case["cols"] = _log_int(rng, 32, side), _log_int(rng, 32, side)
    else:
        case["n"] = _log_int(rng, 1000, min(top, 1 << 22 if kind == "rmat" else 1 << 24))
        case["m"] = int(case["n"] * rng.uniform(4.0, 16.0))
    return case


# ---------------------------------------------------------------------------
# inputs


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _offsets(src, n):
    row_off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(src, minlength=n), 0, out=row_off[1:])
    return row_off


def _gnm(n, m, wmax, gen):
    """Directed G(n, m): endpoints uniform, no self-loops, duplicates kept."""
    row_off = _offsets(torch.randint(n, (m,), device="cuda", dtype=torch.int32, generator=gen), n)
    src = torch.repeat_interleave(torch.arange(n, dtype=torch.int32, device="cuda"), row_off.diff(), output_size=m)
    col = torch.randint(n - 1, (m,), device="cuda", dtype=torch.int32, generator=gen)
    col += col >= src
    w = torch.randint(wmax, (m,), device="cuda", dtype=torch.int32, generator=gen)
    return row_off, col, w


def _rmat(n, m, wmax, gen):
    """R-MAT (.57, .19, .19, .05), self-loops and duplicates kept; an n that is
    no power of two scales the drawn vertices down to it."""
    scale = (n - 1).bit_length()
    src = torch.zeros(m, dtype=torch.int32, device="cuda")
    col = torch.zeros(m, dtype=torch.int32, device="cuda")
    for _ in range(scale):
        u = torch.rand(m, device="cuda", generator=gen)
        down = u >= 0.76
        right = ((u >= 0.57) & (u < 0.76)) | (u >= 0.95)
        src.mul_(2).add_(down)
        col.mul_(2).add_(right)
    if n != 1 << scale:
        src = ((src.long() * n) >> scale).int()
        col = ((col.long() * n) >> scale).int()
    src, order = torch.sort(src)
    return _offsets(src, n), col[order], torch.randint(wmax, (m,), device="cuda", dtype=torch.int32, generator=gen)


def _grid(rows, cols, wmax, gen):
    """4-neighbour grid, one weight in [1, wmax) per undirected edge."""
    n = rows * cols
    v = torch.arange(n, device="cuda").view(rows, cols)
    across = torch.randint(1, wmax, (rows, cols), device="cuda", generator=gen)  # edge (r, c)-(r, c+1)
    along = torch.randint(1, wmax, (rows, cols), device="cuda", generator=gen)  # edge (r, c)-(r+1, c)
    pairs = [(v[:, :-1], v[:, 1:], across[:, :-1]), (v[:-1], v[1:], along[:-1])]
    src = torch.cat([x.reshape(-1) for a, b, _ in pairs for x in (a, b)])
    col = torch.cat([x.reshape(-1) for a, b, _ in pairs for x in (b, a)])
    w = torch.cat([c.reshape(-1) for _, _, c in pairs for _ in (0, 1)])
    src, order = torch.sort(src, stable=True)
    return _offsets(src, n), col[order].int(), w[order].int()


def _vertices(case):
    return case["rows"] * case["cols"] if case["graph"] == "grid" else case["n"]


def _csr(case, gen):
    if case["graph"] == "grid":
        return _grid(case["rows"], case["cols"], case["wmax"], gen)
    make = _gnm if case["graph"] == "gnm" else _rmat
    return make(case["n"], case["m"], case["wmax"], gen)


def _source(case, row_off, gen):
    """One source as the study takes it: a grid's corner, a power-law graph's
    hub, a random vertex of a uniform graph."""
    if case["graph"] == "grid":
        return 0
    if case["graph"] == "rmat":
        return int(row_off.diff().argmax())
    return int(torch.randint(case["n"], (1,), device="cuda", generator=gen))


def _sources(case, row_off, gen):
    """Several sources: random vertices that have out-edges."""
    has = (row_off.diff() > 0).nonzero().view(-1)
    return [int(x) for x in has[torch.randint(has.numel(), (case["sources"],), device="cuda", generator=gen)].tolist()]


def _uneven(case, seed):
    """(n, m, seed, sources) of the graphs of an uneven batch: n log-uniform,
    average degree uniform in [4, 32] (the sizes belong to the case, the edges
    and sources to the seed)."""
    rng = np.random.default_rng(case["graphs"])
    n = np.exp2(rng.uniform(math.log2(case["nmin"]), math.log2(case["nmax"]), case["graphs"])).astype(np.int64)
    m = np.rint(n * rng.uniform(4.0, 32.0, case["graphs"])).astype(np.int64)
    rng = np.random.default_rng(seed)
    return [(int(a), int(b), int(seed) * 1000 + i, [int(s) for s in rng.integers(0, a, case["sources"])])
            for i, (a, b) in enumerate(zip(n, m))]


def _policy_weights():
    """A policy network in hand: IN-SIMPLE phases (arm 2) while the fringe has
    fewer than about 1500 vertices, IN-STATIC on the sparse queue otherwise."""
    w1, w2, w3 = np.zeros((8, 32), np.float32), np.eye(32, dtype=np.float32), np.zeros((32, 4), np.float32)
    w1[:, :8] = np.eye(8, dtype=np.float32)
    w3[0, 2] = 6.0  # log2(1 + |F|) / 4
    zero = np.zeros(32, np.float32)
    return np.concatenate([w1.ravel(), zero, w2.ravel(), zero, w3.ravel(), np.float32([0.0, 1.0, -3.0, 1.0])])


def _training_set(case, seed):
    """Weights and samples with the ranges of the policy's features (fringe,
    settled and relaxed counts on log scales) and of its targets (log2 of the
    nanoseconds per settled vertex)."""
    gen = _generator(seed)
    b = case["batch"]
    x = torch.rand(b, 8, device="cuda", generator=gen)
    x[:, 1] = x[:, 1] ** 4 * 0.5
    target = 2.0 + 12.0 * torch.rand(b, device="cuda", generator=gen)
    arm = torch.randint(4, (b,), device="cuda", dtype=torch.int32, generator=gen)
    lim = torch.full((sp.POLICY_WEIGHTS,), math.sqrt(6.0 / 32), device="cuda")
    w = (2.0 * torch.rand(sp.POLICY_WEIGHTS, device="cuda", generator=gen) - 1.0) * lim
    return w, x, target, arm


def _batch(call, graphs, sources, crit):
    """A prepared batch whose distance arrays lie one after another in one buffer."""
    sizes = [g.n for g in graphs]
    dist = torch.empty(sum(sizes), dtype=torch.int64, device="cuda")
    return {"call": call, "batch": sp.Batch(graphs, sources, crit, outs=list(dist.split(sizes))), "dist": dist}


def prepare(case, seed):
    call = case["call"]
    if call == "train":
        w, x, target, arm = _training_set(case, seed)
        return {"call": call, "w0": w, "x": x, "target": target, "arm": arm, "w": torch.empty_like(w),
                "m1": torch.empty_like(w), "m2": torch.empty_like(w), "grad": torch.empty_like(w),
                "loss": torch.empty(1, device="cuda")}
    crit = CRITERIA[case["criterion"]]
    reverse = case["criterion"] != "in_out"
    if call == "uneven":
        graphs, sources = [], []
        for n, m, gseed, src in _uneven(case, seed):
            g = sp.Graph(n, *_gnm(n, m, case["wmax"], _generator(gseed)), reverse=reverse)
            graphs += [g] * len(src)
            sources += src
        return _batch(call, graphs, sources, crit)
    gen = _generator(seed)
    n = _vertices(case)
    row_off, col, w = _csr(case, gen)
    if call == "create":
        host = [t.cpu().pin_memory().numpy().view(d) for t, d in ((row_off, np.uint64), (col, np.uint32), (w, np.uint32))]
        out = torch.empty(n, dtype=torch.int64, pin_memory=True).numpy().view(np.uint64)
        return {"call": call, "n": n, "host": host, "source": _source(case, row_off, gen), "criterion": crit, "out": out}
    graph = sp.Graph(n, row_off, col, w, reverse=reverse)
    if call == "batch":
        if case["criterion"] == "learned":
            sp.policy_load(_policy_weights())
        return _batch(call, [graph] * case["sources"], _sources(case, row_off, gen), crit)
    return {"call": call, "graph": graph, "source": _source(case, row_off, gen), "criterion": crit,
            "out": torch.empty(n, dtype=torch.int64, device="cuda")}


def run(state):
    call = state["call"]
    if call == "solve":
        dist, phases = sp.solve(state["graph"], state["source"], state["criterion"], out=state["out"])
        return {"dist": dist, "phases": phases}
    if call in ("batch", "uneven"):
        state["batch"].launch()
        return {"dist": state["dist"], "phases": state["batch"].phases}
    if call == "create":
        graph = sp.Graph(state["n"], *state["host"])
        dist, phases = sp.solve(graph, state["source"], state["criterion"], out=state["out"])
        graph.close()
        return {"dist": dist, "phases": phases}
    w, m1, m2 = state["w"], state["m1"], state["m2"]
    w.copy_(state["w0"])  # a step from the same weights every time
    m1.zero_()
    m2.zero_()
    grad, loss = sp.mlp_backward(w, state["x"], state["target"], state["arm"], grad=state["grad"], loss=state["loss"])
    sp.mlp_adam(w, grad, m1, m2, 1e-2, 1)
    return {"grad": grad, "loss": loss, "w": w, "m1": m1, "m2": m2}


def work(case):
    """Each input read once, each output written once; an addition and a
    comparison per edge (two multiply-adds per weight and direction for the
    network)."""
    if case["call"] == "train":
        b, p = case["batch"], sp.POLICY_WEIGHTS
        return {"bytes": b * (8 + 1 + 1) * 4 + p * 4 * 8, "flops": 6 * b * p}
    if case["call"] == "uneven":
        n, m, solves = 0, 0, case["sources"]
        spec = _uneven(case, 0)
        n, m = sum(s[0] for s in spec), sum(s[1] for s in spec)
    else:
        n, solves = _vertices(case), case.get("sources", 1)
        m = 4 * n - 2 * (case["rows"] + case["cols"]) if case["graph"] == "grid" else case["m"]
    # edges {target, cost} and row offsets, static minima, distances of every solve
    return {"bytes": 8 * m + 8 * n + 8 * n + 8 * n * solves, "flops": 2 * m * solves}


# ---------------------------------------------------------------------------
# the same outputs in plain torch


def _distances(row_off, col, w, sources):
    """Shortest distances by rounds of relaxations over all edges (-1: unreachable)."""
    n, far = row_off.numel() - 1, 1 << 62
    src = torch.repeat_interleave(torch.arange(n, device="cuda"), row_off.diff(), output_size=col.numel())
    col, w = col.long(), w.long()
    out = []
    for s in sources:
        d = torch.full((n,), far, dtype=torch.int64, device="cuda")
        d[s] = 0
        while True:
            before = d.clone()
            for _ in range(8):
                d.scatter_reduce_(0, col, d[src] + w, "amin")
            if torch.equal(d, before):
                break
        out.append(torch.where(d >= far, -1, d))
    return out


def exact(case, seed):
    call = case["call"]
    if call == "train":
        w, x, target, arm = (t.double() if t.is_floating_point() else t.long() for t in _training_set(case, seed))
        w.requires_grad_(True)
        w1, b1, w2, b2, w3, b3 = torch.split(w, [256, 32, 1024, 32, 128, 4])
        h = torch.relu(x @ w1.view(8, 32) + b1)
        h = torch.relu(h @ w2.view(32, 32) + b2)
        y = (h @ w3.view(32, 4) + b3).gather(1, arm[:, None])[:, 0]
        loss = ((y - target) ** 2).mean()
        (grad,) = torch.autograd.grad(loss, w)
        w = w.detach()
        # Adam's first step from zero moments (both bias corrections cancel the decay factors), with
        # the rates and factors as the single-precision values that the call takes
        lr, eps, beta1, beta2 = (float(np.float32(v)) for v in (1e-2, 1e-8, 0.9, 0.999))
        return {"grad": grad, "loss": loss.detach().view(1), "w": w - lr * grad / (grad.abs() + eps),
                "m1": (1.0 - beta1) * grad, "m2": (1.0 - beta2) * grad ** 2}
    if call == "uneven":
        out = []
        for n, m, gseed, src in _uneven(case, seed):
            out += _distances(*_gnm(n, m, case["wmax"], _generator(gseed)), src)
        return {"dist": torch.cat(out), "phases": None}
    if call == "batch" and _vertices(case) * case["sources"] > 1 << 25:
        return None  # minutes of relaxation rounds
    gen = _generator(seed)
    row_off, col, w = _csr(case, gen)
    if call == "batch":
        return {"dist": torch.cat(_distances(row_off, col, w, _sources(case, row_off, gen))), "phases": None}
    (dist,) = _distances(row_off, col, w, [_source(case, row_off, gen)])
    return {"dist": dist.cpu().numpy().view(np.uint64) if call == "create" else dist, "phases": None}
