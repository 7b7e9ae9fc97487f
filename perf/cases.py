"""The work a user of this framework has it do, as cases that can be timed.

A pass is a whole call sequence through the public entry points, as a user's
program makes it for graphs it has on the device: load the CSR (checked),
compute, free the handle.  Nothing computed for one pass serves the next: the
context (stream, options, workspace, model weights) is what a program keeps.

Graphs have the shapes of the paper's networks: Barabasi-Albert (undirected,
collaboration-like), R-MAT (directed, web- and social-network-like),
Erdos-Renyi (directed, no hubs) and street grids with missing edges.
"""
import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from paper_1704_01077_gb300 import graphgen as gg
from paper_1704_01077_gb300 import tkc, train_order

DEG, NB, LEARNED_NB = tkc.TKC_ORDER_DEG, tkc.TKC_ORDER_NB, tkc.TKC_ORDER_LEARNED_NB


def listed():
    return [
        # the smallest call: the library's defaults (degree order) on a graph of 2 000 vertices; launches and waits count
        {"name": "ba2k_deg", "do": "topk", "graph": "ba", "n": 2000, "m": 4, "order": DEG, "k": 10},
        # a small directed graph and the single most central vertex, neighbourhood-bound order
        {"name": "er5k_nb_k1", "do": "topk", "graph": "er", "n": 5001, "m": 8, "order": NB, "k": 1},
        # an ordinary social network, the fast order (NBCut)
        {"name": "rmat16_nb", "do": "topk", "graph": "rmat", "scale": 16, "m": 16, "order": NB, "k": 10},
        # the same with the default order (DegCut), which examines every source
        {"name": "rmat16_deg", "do": "topk", "graph": "rmat", "scale": 16, "m": 16, "order": DEG, "k": 10},
        # a collaboration network of a million vertices, a long list
        {"name": "ba1m_nb_k100", "do": "topk", "graph": "ba", "n": 1000000, "m": 5, "order": NB, "k": 100},
        # a large network with the default order
        {"name": "rmat20_deg", "do": "topk", "graph": "rmat", "scale": 20, "m": 16, "order": DEG, "k": 10},
        # harmonic centrality of a large network
        {"name": "rmat20_harmonic", "do": "harmonic", "graph": "rmat", "scale": 20, "m": 16, "order": NB, "k": 10},
        # the largest network: 4.2 million vertices, 65 million arcs
        {"name": "rmat22_nb", "do": "topk", "graph": "rmat", "scale": 22, "m": 16, "order": NB, "k": 10},
        # many graphs of uneven sizes in one launch, half undirected and half directed
        {"name": "multi512_nb", "do": "multi", "graphs": 512, "lo": 1000, "hi": 200000, "order": NB, "k": 10},
        # a street network (long paths), by level bounds (NBBound)
        {"name": "grid_bound", "do": "bound", "graph": "grid", "rows": 301, "cols": 299, "order": NB, "k": 10},
        # exact farness of half a graph's vertices: targets the source-order model is trained on
        {"name": "sums_rmat14", "do": "sums", "graph": "rmat", "scale": 14, "m": 16},
        # the model's backward pass on a training batch
        {"name": "mlp_gradient", "do": "gradient", "m": 2048},
    ]


def _log(rng, lo, hi):
    return min(int(hi), max(int(lo), int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["topk", "topk", "topk", "topk", "harmonic", "learned", "multi", "bound", "sums", "gradient",
                       "forward"])
    if kind == "gradient":
        return {"do": "gradient", "m": _log(rng, 1, 8192)}
    if kind == "forward":
        return {"do": "forward", "m": _log(rng, 1, 1 << 21)}
    if kind == "multi":
        return {"do": "multi", "graphs": _log(rng, 2, 200), "lo": _log(rng, 50, 2000), "hi": _log(rng, 3000, 200000),
                "order": rng.choice([DEG, NB]) if rng.random() < 0.3 else NB, "k": _log(rng, 1, 50)}
    if kind == "bound":
        rows = _log(rng, 20, 300)
        return {"do": "bound", "graph": "grid", "rows": rows, "cols": _log(rng, 20, 300), "order": rng.choice([DEG, NB]),
                "k": _log(rng, 1, 50)}
    if kind == "sums":
        if rng.random() < 0.5:
            return {"do": "sums", "graph": "rmat", "scale": rng.randint(9, 14), "m": 16}
        return {"do": "sums", "graph": "ba", "n": _log(rng, 500, 20000), "m": rng.randint(2, 6)}
    if kind == "learned":
        return {"do": "topk", "graph": "rmat", "scale": rng.randint(12, 18), "m": 16, "order": LEARNED_NB,
                "k": _log(rng, 1, 20)}
    case = {"do": kind, "order": rng.choice([DEG, NB]), "k": _log(rng, 1, 200)}
    top = 300000 if case["order"] == DEG else 1000000
    g = rng.choice(["ba", "er", "rmat", "rmat"])
    if g == "rmat":
        return {**case, "graph": g, "scale": rng.randint(10, 18 if case["order"] == DEG else 21), "m": rng.randint(8, 16)}
    if g == "er":
        return {**case, "graph": g, "n": _log(rng, 1000, min(top, 200000)), "m": rng.randint(6, 12)}
    return {**case, "graph": g, "n": _log(rng, 1000, top), "m": rng.randint(2, 6)}


# ---------------------------------------------------------------------- inputs


def _csr_from_keys(key, n):
    """Sorted distinct (source * n + target) -> CSR (offsets, cols) on the device."""
    src = torch.div(key, n, rounding_mode="floor")
    cols = (key - src * n).to(torch.int32)
    bounds = torch.searchsorted(src, torch.arange(n + 1, device=key.device, dtype=src.dtype))
    return bounds.to(torch.int32).contiguous(), cols.contiguous()


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed & 0x7fffffffffffffff)


def _rmat(scale, m, seed):
    """R-MAT, a/b/c/d = 0.57/0.19/0.19/0.05, self-loops and duplicates removed, ids permuted."""
    n, gen = 1 << scale, _generator(seed)
    src = torch.zeros(m * n, dtype=torch.int64, device="cuda")
    dst = torch.zeros_like(src)
    for _ in range(scale):
        u = torch.rand(m * n, generator=gen, device="cuda")
        src = 2 * src + (u >= 0.76)
        dst = 2 * dst + (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
    perm = torch.randperm(n, generator=gen, device="cuda")
    src, dst = perm[src], perm[dst]
    key = torch.unique((src * n + dst)[src != dst])
    return n, *_csr_from_keys(key, n), True


def _er(n, m, seed):
    gen = _generator(seed)
    src = torch.randint(n, (m * n,), generator=gen, device="cuda")
    dst = torch.randint(n, (m * n,), generator=gen, device="cuda")
    key = torch.unique((src * n + dst)[src != dst])
    return n, *_csr_from_keys(key, n), True


def _to_device(g):
    return g.n, torch.from_numpy(g.offsets.view(np.int32)).cuda(), torch.from_numpy(g.cols.view(np.int32)).cuda(), \
        g.directed


def _graph(case, seed):
    kind = case["graph"]
    if kind == "rmat":
        return _rmat(case["scale"], case["m"], seed)
    if kind == "er":
        return _er(case["n"], case["m"], seed)
    if kind == "grid":
        return _to_device(gg.grid(case["rows"], case["cols"], seed=seed & 0x7fffffff, drop=0.1))
    return _to_device(gg.barabasi_albert(case["n"], case["m"], gg.splitmix64(seed)))


def _sizes(case):
    """Vertex counts of a multi-graph case (the same for every seed: they are its size)."""
    return gg.log_uniform_sizes(case["graphs"], case["lo"], case["hi"], gg.workload_seed(3))


def _many(case, seed):
    sizes = _sizes(case)
    with ThreadPoolExecutor(8) as pool:
        ba = {i: pool.submit(gg.barabasi_albert, n, 4, gg.splitmix64(seed + i)) for i, n in enumerate(sizes) if i % 2 == 0}
        er = {i: _er(n, 8, seed + i) for i, n in enumerate(sizes) if i % 2 == 1}
        return [er[i] if i in er else _to_device(ba[i].result()) for i in range(len(sizes))]


def _model(seed):
    """He-uniform weights and zero biases in the library's parameter layout."""
    rng = np.random.default_rng(seed)
    w = np.zeros(tkc.TKC_MLP_PARAMS, np.float32)
    w[:320] = rng.uniform(-1, 1, 320) * math.sqrt(6 / 5)
    w[384:4480] = rng.uniform(-1, 1, 4096) * math.sqrt(6 / 64)
    w[4544:4608] = rng.uniform(-1, 1, 64) * math.sqrt(6 / 64)
    return w


def _samples(case, seed):
    gen = _generator(seed)
    x = torch.randn(case["m"], tkc.TKC_MLP_FEATURES, generator=gen, device="cuda")
    t = torch.randn(case["m"], generator=gen, device="cuda")
    return x, t


def _sources(graph):
    """n/2 vertices that reach another one, in id order."""
    return torch.nonzero(graph[1].diff() > 0).flatten()[:graph[0] // 2]


class State:
    """A context and the inputs; the context goes with the state."""

    def __init__(self, case, seed):
        self.case = case
        self.options = tkc.Options(order=case.get("order", DEG))
        if self.options.order == LEARNED_NB:
            self.options.seed_factor = 5
        self.ctx = tkc.tkc_create(self.options)
        if case["do"] in ("gradient", "forward"):
            tkc.tkc_set_source_model(self.ctx, _model(seed))
            self.x, self.t = _samples(case, seed)
            self.grad = torch.zeros(tkc.TKC_MLP_PARAMS, device="cuda")
            self.y = torch.zeros(case["m"], device="cuda")
        elif case["do"] == "multi":
            self.graphs = _many(case, seed)
        else:
            self.graph = _graph(case, seed)
            if self.options.order == LEARNED_NB:
                tkc.tkc_set_source_model(self.ctx, train_order.load_weights())
            if case["do"] == "sums":
                self.sources = _sources(self.graph).cpu().numpy().astype(np.uint32)

    def __del__(self):
        if getattr(self, "ctx", None):
            tkc.tkc_destroy(self.ctx)
            self.ctx = None


def prepare(case, seed):
    return State(case, seed)


# ---------------------------------------------------------------------- a pass


def _entries(r):
    return {"ids": r.ids, "dist_sum": r.dist_sum, "reach": r.reach, "farness": r.farness, "closeness": r.closeness,
            "tied": r.n_tied_at_kth}


def run(state):
    case = state.case
    do = case["do"]
    if do == "gradient":
        loss = tkc.tkc_mlp_gradient(state.ctx, state.x, state.t, state.grad)
        return {"grad": state.grad, "loss": np.float32(loss)}
    if do == "forward":
        tkc.tkc_mlp_forward(state.ctx, state.x, state.y)
        return {"y": state.y}
    if do == "multi":
        handles = tkc.tkc_load_csr_many(state.ctx, state.graphs)
        try:
            results = [_entries(r) for r in tkc.tkc_topk_closeness_multi(state.ctx, handles, case["k"])]
        finally:
            for h in handles:
                tkc.tkc_free_graph(h)
        return {key: np.concatenate([np.atleast_1d(r[key]) for r in results]) for key in results[0]}
    h = tkc.tkc_load_csr(state.ctx, *state.graph)
    try:
        if do == "sums":
            S, r = tkc.tkc_distance_sums(h, state.sources)
            return {"dist_sum": S, "reach": r}
        call = {"topk": tkc.tkc_topk_closeness, "harmonic": tkc.tkc_topk_harmonic, "bound": tkc.tkc_topk_closeness_bound}
        return _entries(call[do](h, case["k"]))
    finally:
        tkc.tkc_free_graph(h)


# ---------------------------------------------------------------------- what a pass cannot do without


def _shape(case):
    """(vertices, arcs) a case's graphs hold, about (duplicates aside)."""
    if case["do"] == "multi":
        sizes = _sizes(case)
        return sum(sizes), sum(8 * n for n in sizes)
    if case["graph"] == "rmat":
        return 1 << case["scale"], case["m"] << case["scale"]
    if case["graph"] == "grid":
        n = case["rows"] * case["cols"]
        return n, int(3.6 * n)
    return case["n"], case["m"] * case["n"] * (1 if case["graph"] == "er" else 2)


def work(case):
    """Inputs read once, outputs written once.  Sums of distances also need
    every (source, vertex) pair once, one bit each."""
    p = tkc.TKC_MLP_PARAMS
    if case["do"] in ("gradient", "forward"):
        m, layers = case["m"], 2 * (5 * 64 + 64 * 64 + 64)
        if case["do"] == "forward":
            return {"bytes": 4 * m * 6 + 2 * p, "flops": m * layers}
        return {"bytes": 4 * m * 6 + 2 * p + 4 * p, "flops": 3 * m * layers}
    n, arcs = _shape(case)
    size = 4 * (n + 1) + 4 * arcs
    if case["do"] == "sums":
        return {"bytes": size + 6 * n + n * n // 16, "flops": 0}
    return {"bytes": size + 32 * case["k"] * case.get("graphs", 1), "flops": 0}


# ---------------------------------------------------------------------- the same by other means, in 64 bits


def _dense_levels(graph, columns):
    """Level by level BFS from `columns` (source ids) by products with the dense
    adjacency matrix: yields (d, members of level d per source) as 0/1 columns."""
    n, off, cols, _ = graph
    src = torch.repeat_interleave(torch.arange(n, device="cuda"), off.diff().long())
    adj = torch.zeros(n, n, dtype=torch.float16, device="cuda")
    adj[cols.long(), src] = 1
    front = torch.zeros(n, len(columns), dtype=torch.float16, device="cuda")
    front[columns, torch.arange(len(columns), device="cuda")] = 1
    seen = front > 0
    d = 0
    while True:
        d += 1
        new = (adj @ front > 0) & ~seen
        if not bool(new.any()):
            return
        yield d, new
        seen |= new
        front = new.to(torch.float16)


def _all_sums(graph, columns, harmonic=False):
    S = torch.zeros(len(columns), dtype=torch.float64 if harmonic else torch.int64, device="cuda")
    r = torch.ones(len(columns), dtype=torch.int64, device="cuda")
    for b in range(0, len(columns), 8192):
        part = columns[b:b + 8192]
        for d, new in _dense_levels(graph, part):
            c = new.sum(0)
            S[b:b + len(part)] += c.double() / d if harmonic else c * d
            r[b:b + len(part)] += c
    return S, r


def _exact_top(case, graph):
    n = graph[0]
    S, r = _all_sums(graph, torch.arange(n, device="cuda"), case["do"] == "harmonic")
    S, r = S.cpu().numpy(), r.cpu().numpy()
    with np.errstate(divide="ignore"):
        if case["do"] == "harmonic":
            c = S
            f = 1 / c
        else:
            num, den = (n - 1) * S.astype(np.float64), (r - 1).astype(np.float64) ** 2
            f = np.where(r > 1, num / np.where(r > 1, den, 1), np.inf)
            c = np.where(r > 1, den / np.where(r > 1, num, 1), 0)
    top = np.lexsort((np.arange(n), f))[:case["k"]]
    return {"ids": top.astype(np.uint32), "dist_sum": (S[top] * (case["do"] != "harmonic")).astype(np.uint64),
            "reach": r[top].astype(np.uint32), "farness": f[top], "closeness": c[top], "tied": int((f == f[top[-1]]).sum())}


def _exact_model(case, seed):
    w = torch.from_numpy(_model(seed)).to(torch.bfloat16).double().cuda()
    x, t = _samples(case, seed)
    w.requires_grad_(True)
    h = torch.relu(x.double() @ w[:320].view(64, 5).T + w[320:384])
    h = torch.relu(h @ w[384:4480].view(64, 64).T + w[4480:4544])
    y = h @ w[4544:4608] + w[4608]
    if case["do"] == "forward":
        return {"y": y.detach()}
    loss = ((y - t.double()) ** 2).mean()
    loss.backward()
    return {"grad": w.grad, "loss": float(loss)}


def exact(case, seed):
    if case["do"] in ("gradient", "forward"):
        return _exact_model(case, seed)
    if case["do"] in ("multi", "bound") or _shape(case)[0] > 16384:
        return None  # every pair of a large or deep graph takes too long this way
    graph = _graph(case, seed)
    if case["do"] == "sums":
        S, r = _all_sums(graph, _sources(graph))
        return {"dist_sum": S.cpu().numpy().astype(np.uint64), "reach": r.cpu().numpy().astype(np.uint32)}
    return _exact_top(case, graph)
