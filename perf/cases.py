"""The workloads this library is timed on: calls a user's program makes through the Python
binding, from the one-time graph steps (CSR build, block partition, locality layout, Trishla
prune and compaction) to the solves (one small graph, many sources on a large one, a
high-diameter grid, a batch of small problems, a warm start) and the gradient.

`listed()` names the fixed ones, `draw(rng)` gives more of the same ranges, `prepare` makes
what a program holds before the call, `run` is one pass, `work` the bytes and additions a pass
cannot do without, and `exact` the same outputs from plain torch in 64 bits.

Sizes are those of the repository's workloads: the Erdos-Renyi graph of 16,384 vertices, R-MAT
scale 22 (edge factor 16, 148 partitions, 8 sources), the 4096 x 4096 grid, 512 small graphs
with 16 sources each, and R-MAT scale 18 with 32 float32 sources.  Schedules are the ones the
autotuner picks on them.
"""
import math

import numpy as np
import torch

import paper_2103_12012_gb300 as sssp

NONE = 0xFFFFFFFF
INF = 0xFFFFFFFF


# ------------------------------------------------------------------------------- cases

def listed():
    return [
        # a program that ingests a small graph: launches and latency count
        dict(name="build_er16k", kind="build", graph="er", V=16384, E=131072, distinct=130000, wtype="u32", P=4),
        # ingest of a large edge list (with duplicates and loops)
        dict(name="build_rmat22", kind="build", graph="rmat", V=1 << 22, E=1 << 26, distinct=65000000, wtype="u32",
             P=148),
        # the one-time renumbering before many solves on that graph
        dict(name="layout_rmat22", kind="layout", graph="rmat", V=1 << 22, E=1 << 26, distinct=65000000, wtype="u32",
             P=148),
        # prune of a large graph in the paper's local mode
        dict(name="prune_rmat21_local", kind="prune", graph="rmat", V=1 << 21, E=1 << 25, distinct=32000000,
             wtype="u32", P=148, mode=0),
        # prune with any witness on a small float32 graph of odd size
        dict(name="prune_rmat16_global_f32", kind="prune", graph="rmat", V=60013, E=16 * 60013, distinct=800001,
             wtype="f32", P=4, mode=1),
        # the graph without its pruned edges (the share that the prune drops there), with the block
        # bounds and inter-edge counts (the message threshold of the termination rule) of what is left
        dict(name="compact_rmat22", kind="compact", graph="rmat", V=1 << 22, E=1 << 26, distinct=65000000,
             wtype="u32", P=148, pruned=0.04),
        # one query on a small graph, the call a program makes without tuning anything
        dict(name="solve_er16k", kind="solve", graph="er", V=16384, E=131072, distinct=130000, wtype="u32", P=4, S=1,
             layout=False, delta=0.0, tile=0, split=0, hubs=0, policy="relative"),
        # many sources on a large low-diameter graph (tuned schedule on the layout graph)
        dict(name="solve_rmat22_8src", kind="solve", graph="rmat", V=1 << 22, E=1 << 26, distinct=65000000, wtype="u32", P=148, S=8,
             layout=True, delta=10.0, tile=1024, split=1, hubs=256, policy="relative"),
        # a road-like network: thousands of hops from a corner
        dict(name="solve_grid4096", kind="solve", graph="grid", rows=4096, cols=4096, wtype="u32", P=148, S=1,
             layout=False, delta=2982.0, tile=1024, split=4, hubs=0, policy="relative"),
        # many independent small problems of uneven size in one graph-captured launch
        dict(name="batch_512x16", kind="batch", graphs=512, lo=10.0, hi=17.0, S=16, wtype="u32", threads=1024,
             tile=2048, delta=16.0),
        # a training step through shortest paths: distances, then the gradient of the weights
        dict(name="grad_rmat18_f32", kind="grad", graph="rmat", V=1 << 18, E=1 << 21, distinct=1950000, wtype="f32", P=16, S=32,
             delta=0.62, tile=2048),
        # a new result after a thousandth of the weights fell (odd vertex count)
        dict(name="update_rmat20", kind="update", graph="rmat", V=1000003, E=16 * 1000003, distinct=15000000, wtype="u32", P=148,
             S=4, layout=True, delta=10.0, tile=1024, split=1, hubs=256, policy="relative", changed=0.001),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sized(rng, graph, lo, hi, factors=(8, 16)):
    V = _log_int(rng, lo, hi)
    E = V * rng.choice(factors) - rng.randrange(0, 8)
    return dict(graph=graph, V=V, E=E, distinct=int(E * rng.uniform(0.7, 0.95 if graph == "er" else 0.75)))


def draw(rng):
    kind = rng.choice(["build", "build", "layout", "compact", "prune", "solve", "solve", "solve", "batch", "grad",
                       "update"])
    wtype = rng.choice(["u32", "f32"])
    if kind in ("build", "layout", "compact"):
        c = _sized(rng, rng.choice(["er", "rmat"]), 1 << 10, 1 << 22)
        c.update(kind=kind, wtype=wtype, P=_log_int(rng, 1, 148))
        if kind == "compact":
            c["pruned"] = rng.choice([0.0, 0.001, 0.04, 0.3])
        return c
    if kind == "prune":
        mode = rng.randrange(2)
        c = _sized(rng, "rmat", 1 << 13, 1 << 16 if mode else 1 << 21)  # (few triangles in er)
        c.update(kind=kind, wtype=wtype, P=rng.randint(64, 148) if mode == 0 else rng.randint(1, 148), mode=mode)
        return c
    if kind == "solve":
        graph = rng.choice(["er", "rmat", "grid"])
        scale = 1.0 if wtype == "u32" else 1.25 / 128.0  # float32 weights average 1.25, uint32 ones 128
        c = dict(kind=kind, graph=graph, wtype=wtype, P=rng.randint(4, 148), S=rng.randint(1, 8), layout=False,
                 tile=rng.choice([1024, 2048]), split=1, hubs=0, policy=rng.choice(["relative", "relative", "fixed"]))
        if graph == "grid":
            c.update(rows=_log_int(rng, 64, 4096), cols=_log_int(rng, 64, 4096), S=1, split=rng.choice([1, 4]),
                     delta=2982.0 if wtype == "u32" else 5.0, policy="relative")
        else:
            c.update(_sized(rng, graph, 1 << 12, 1 << 22))
            if graph == "rmat" and rng.random() < 0.7:
                c.update(layout=True, hubs=rng.choice([0, 256]))
            c["delta"] = rng.choice([5.0, 10.0, 16.0]) * scale
        return c
    if kind == "batch":
        hi = rng.uniform(11.0, 17.0)
        return dict(kind=kind, graphs=_log_int(rng, 8, 512), lo=10.0, hi=hi, S=rng.randint(1, 16), wtype=wtype,
                    threads=rng.choice([512, 1024]), tile=rng.choice([1024, 2048]),
                    delta=16.0 if wtype == "u32" else 0.16)
    if kind == "grad":
        c = _sized(rng, rng.choice(["er", "rmat"]), 1 << 12, 1 << 18, factors=(8,))
        c.update(kind=kind, wtype="f32", P=rng.randint(1, 64), S=rng.randint(1, 32), delta=0.62, tile=2048)
        return c
    c = _sized(rng, "rmat", 1 << 14, 1 << 21, factors=(16,))
    c.update(kind=kind, wtype=wtype, P=rng.randint(16, 148), S=rng.randint(1, 8), layout=rng.random() < 0.5,
             delta=10.0 if wtype == "u32" else 0.1, tile=1024, split=1, hubs=0, policy="relative",
             changed=rng.choice([0.0001, 0.001, 0.01]))
    return c


# ------------------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
    return g


def _weights(n, wtype, gen, hi=255):
    if wtype == "u32":
        return torch.randint(1, hi + 1, (n,), generator=gen, device="cuda", dtype=torch.int32)
    # uniform on [0.5, 2) plus a jitter that makes shortest paths unique
    return 0.5 + 1.5 * torch.rand(n, generator=gen, device="cuda") + 1e-4 * torch.rand(n, generator=gen, device="cuda")


def _er(V, E, gen):
    src = torch.randint(0, V, (E,), generator=gen, device="cuda", dtype=torch.int32)
    dst = torch.randint(0, V, (E,), generator=gen, device="cuda", dtype=torch.int32)
    return src, dst


def _rmat(V, E, gen):
    """R-MAT (.57, .19, .19, .05) with permuted vertex ids; duplicates and loops stay."""
    src = torch.zeros(E, dtype=torch.int32, device="cuda")
    dst = torch.zeros(E, dtype=torch.int32, device="cuda")
    for _ in range(max(1, (V - 1).bit_length())):
        r = torch.rand(E, generator=gen, device="cuda")
        src = src * 2 + (r >= 0.76).int()
        dst = dst * 2 + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95)).int()
    perm = torch.randperm(V, generator=gen, device="cuda").int()
    return perm[(src % V).long()], perm[(dst % V).long()]


def _grid(rows, cols, wtype, gen):
    """4-neighbour grid, both directions of an edge with one weight."""
    ids = torch.arange(rows * cols, dtype=torch.int32, device="cuda").view(rows, cols)
    a = torch.cat([ids[:, :-1].reshape(-1), ids[:-1].reshape(-1)])
    b = torch.cat([ids[:, 1:].reshape(-1), ids[1:].reshape(-1)])
    w = _weights(a.numel(), wtype, gen, hi=1000)
    return torch.cat([a, b]), torch.cat([b, a]), torch.cat([w, w])


def _with_distinct(V, E, distinct, src, dst, more, gen):
    """E edges in random order of which `distinct` pairs differ; the rest repeats them or is loops."""
    def pairs(s, d):
        return torch.unique((s.long() * V + d)[s != d])

    key = pairs(src, dst)
    while key.numel() < distinct:
        key = torch.unique(torch.cat([key, pairs(*more(V, E, gen))]))
    key = key[torch.randperm(key.numel(), generator=gen, device="cuda")[:distinct]]
    loops = torch.randint(0, V, ((E - distinct) // 8,), generator=gen, device="cuda") * (V + 1)
    again = key[torch.randint(0, distinct, (E - distinct - loops.numel(),), generator=gen, device="cuda")]
    key = torch.cat([key, again, loops])[torch.randperm(E, generator=gen, device="cuda")]
    return (key // V).int(), (key % V).int()


def _edges(case, gen):
    """(V, src, dst, w) on the device."""
    if case["graph"] == "grid":
        src, dst, w = _grid(case["rows"], case["cols"], case["wtype"], gen)
        return case["rows"] * case["cols"], src, dst, w
    V, E, more = case["V"], case["E"], _er if case["graph"] == "er" else _rmat
    src, dst = more(V, E, gen)
    if "distinct" in case:
        src, dst = _with_distinct(V, E, case["distinct"], src, dst, more, gen)
    return V, src, dst, _weights(E, case["wtype"], gen)


def _sources(case, V, src, dst, gen):
    """S vertices with an out-edge (the corner of a grid)."""
    if case["graph"] == "grid":
        return torch.zeros(1, dtype=torch.int32, device="cuda")
    tails = src[src != dst]
    pick = torch.randint(0, tails.numel(), (case["S"],), generator=gen, device="cuda")
    return tails[pick].contiguous()


def _options(case):
    return sssp.options(tile=case["tile"], split=case.get("split", 0), delta=case["delta"],
                        policy=sssp.POLICY_NAMES.index(case.get("policy", "relative")), hub_count=case.get("hubs", 0))


def _batch_inputs(case, gen, rng):
    out = []
    n = case["graphs"]
    for i in rng.permutation(n):  # sizes spread evenly over the logarithm, in random order
        V = int(round(2.0 ** (case["lo"] + (case["hi"] - case["lo"]) * (i + 0.5) / n)))
        sub = dict(graph=str(rng.choice(["er", "rmat"])), V=V, E=8 * V, wtype=case["wtype"])
        out.append((_edges(sub, gen), rng.integers(0, V, case["S"]).astype(np.uint32)))
    return out


def _keep(case, E, gen):
    """A prune's keep mask with a fixed number of dropped edges."""
    keep = torch.ones(E, dtype=torch.uint8, device="cuda")
    keep[torch.randperm(E, generator=gen, device="cuda")[:int(E * case["pruned"])]] = 0
    return keep


def _changed(case, w, gen):
    """Indices of the edges whose weight falls, and the weights after."""
    e = torch.randint(0, w.numel(), (max(1, int(w.numel() * case["changed"])),), generator=gen, device="cuda")
    after = w.clone()
    after[e] = w[e] * 0.5 if w.is_floating_point() else (w[e] // 2).clamp(min=1)
    return e, after


def prepare(case, seed):
    gen = _gen(seed)
    kind = case["kind"]
    if kind == "batch":
        graphs, sources = [], []
        for (V, src, dst, w), s in _batch_inputs(case, gen, np.random.default_rng(seed)):
            graphs.append(sssp.build_csr(V, src, dst, w))
            sources.append(s)
        b = sssp.Batch(graphs, sources, sssp.options(threads=case["threads"], tile=case["tile"], delta=case["delta"]))
        b.make_plan()
        return dict(case=case, batch=b)
    V, src, dst, w = _edges(case, gen)
    if kind == "build":
        return dict(case=case, V=V, src=src, dst=dst, w=w)
    g = sssp.build_csr(V, src, dst, w, partitions=case["P"])
    st = dict(case=case, g=g)
    if kind == "compact":
        st["keep"] = _keep(case, g.E, gen)
    if kind in ("solve", "grad", "update"):
        st["sources"] = _sources(case, V, src, dst, gen)
    if kind == "solve":
        if case["layout"]:
            st["g"] = sssp.layout(g)
        st["opts"] = _options(case)
        if case["delta"]:  # a program with a tuned schedule keeps the solver and its workspace
            st["solver"] = sssp.Solver(st["g"], case["S"], st["opts"])
    elif kind == "grad":
        st["opts"] = _options(case)
        st["fn"] = sssp.sssp_function()
        st["w"] = g.w.clone().requires_grad_(True)
        st["grad_dist"] = torch.randn((case["S"], V), generator=gen, device="cuda")
    elif kind == "update":
        if case["layout"]:
            g = st["g"] = sssp.layout(g)
        opts = _options(case)
        st["dist"], st["pred"] = sssp.solve(g, st["sources"], opts)[:2]
        e, w2 = _changed(case, g.w, gen)
        tails = torch.searchsorted(g.row_ptr.long(), e, right=True) - 1
        st["tails"] = (g.ids[tails] if g.ids is not None else tails).int().contiguous()
        g2 = sssp.DeviceGraph(g.V, g.E, g.row_ptr, g.col, w2, g.wtype, g.partitions, g.eid, g.ids, g.slots)
        st["solver"] = sssp.Solver(g2, case["S"], opts)
    return st


# -------------------------------------------------------------------------------- pass

def _graph_out(g):
    return dict(row_ptr=g.row_ptr, col=g.col, w=g.w, eid=g.eid)


def run(st):
    kind = st["case"]["kind"]
    if kind == "build":
        return _graph_out(sssp.build_csr(st["V"], st["src"], st["dst"], st["w"], partitions=st["case"]["P"]))
    if kind == "layout":
        g = sssp.layout(st["g"])
        return dict(_graph_out(g), ids=g.ids, slots=g.slots)
    if kind == "prune":
        keep, witness = sssp.prune(st["g"], mode=st["case"]["mode"])
        return dict(keep=keep, witness=witness)
    if kind == "compact":
        g = sssp.compact(st["g"], st["keep"])
        bounds, inter = sssp.partition(g)
        return dict(_graph_out(g), bounds=bounds, inter=inter)
    if kind == "solve":
        if "solver" in st:
            dist, pred = st["solver"](st["sources"])
        else:
            dist, pred = sssp.solve(st["g"], st["sources"], st["opts"])[:2]
        return dict(dist=dist, pred=pred)
    if kind == "batch":
        st["batch"].replay()
        return dict(dist=st["batch"].dist, pred=st["batch"].pred)
    if kind == "grad":
        dist = st["fn"].apply(st["w"], st["g"], st["sources"], st["opts"])
        (grad_w,) = torch.autograd.grad(dist, st["w"], st["grad_dist"])
        return dict(dist=dist.detach(), grad_w=grad_w)
    # update: the previous result is kept, a copy of it is brought up to date
    dist, pred = st["solver"].update(st["dist"].clone(), st["pred"].clone(), st["tails"])
    return dict(dist=dist, pred=pred)


def work(case):
    """Each input once, each output once; one addition per edge and source."""
    kind = case["kind"]
    if kind == "batch":
        mean_v = (2.0 ** case["hi"] - 2.0 ** case["lo"]) / ((case["hi"] - case["lo"]) * math.log(2.0))
        V = case["graphs"] * mean_v
        E = 8 * V
        return dict(bytes=int(12 * E + 4 * V + 8 * V * case["S"]), flops=int(E * case["S"]))
    if case.get("graph") == "grid":
        V = case["rows"] * case["cols"]
        E = 4 * V - 2 * (case["rows"] + case["cols"])
    else:
        V, E = case["V"], case["E"] if kind == "build" else case["distinct"]
    S = case.get("S", 1)
    if kind == "build":
        return dict(bytes=12 * (E + case["distinct"]) + 4 * V, flops=E)
    if kind == "layout":
        return dict(bytes=20 * E + 16 * V, flops=E)
    if kind == "prune":
        return dict(bytes=13 * E + 4 * V, flops=E)
    if kind == "compact":
        return dict(bytes=21 * E + 8 * V, flops=E)
    if kind == "solve":
        return dict(bytes=8 * E + 4 * V + 8 * S * V, flops=S * E)
    if kind == "grad":
        return dict(bytes=12 * E + 4 * V + 12 * S * V, flops=S * (E + 2 * V))
    return dict(bytes=16 * S * V, flops=int(S * V + 16 * case["changed"] * S * V))


# ------------------------------------------------------------------------------- exact

def _csr64(V, src, dst, w):
    """The canonical CSR: no loops, the least weight of parallel edges (lowest input index on ties)."""
    src, dst = src.long(), dst.long()
    idx = torch.nonzero(src != dst).flatten()
    key = src[idx] * V + dst[idx]
    by_w = torch.sort(w[idx], stable=True).indices
    order = by_w[torch.sort(key[by_w], stable=True).indices]
    key = key[order]
    head = torch.ones_like(key, dtype=torch.bool)
    head[1:] = key[1:] != key[:-1]
    key, eid = key[head], idx[order][head]
    row_ptr = torch.searchsorted(key, torch.arange(V + 1, device="cuda") * V)
    return row_ptr, key // V, key % V, w[eid], eid


def _layout64(V, P, src, dst):
    """ids: inside each block of ceil(V / P) vertices by total degree, highest first, ties by id."""
    B = (V + P - 1) // P
    deg = torch.bincount(src, minlength=V) + torch.bincount(dst, minlength=V)
    ids = torch.sort(deg, descending=True, stable=True).indices
    ids = ids[torch.sort(ids // B, stable=True).indices]
    slots = torch.empty_like(ids)
    slots[ids] = torch.arange(V, device="cuda")
    return ids, slots


def _bellman_ford(V, src, dst, w, source):
    """Least distances in w's type (the fixpoint is unique), inf where unreached."""
    inf = float("inf") if w.is_floating_point() else 1 << 62
    d = torch.full((V,), inf, dtype=w.dtype, device="cuda")
    d[source] = 0
    while True:
        n = d.scatter_reduce(0, dst, torch.where(d[src] < inf, d[src] + w, inf), "amin")
        if torch.equal(n, d):
            return d, inf
        d = n


def _tree(V, src, dst, w, d, inf):
    """Smallest tail of a tight edge into each reached vertex, -1 for the others (and the source)."""
    tight = (d[src] < inf) & (d[src] + w == d[dst])
    p = torch.full((V,), V, dtype=torch.int64, device="cuda")
    p.scatter_reduce_(0, dst[tight], src[tight], "amin")
    return torch.where(p < V, p, -1)


def _solve64(V, src, dst, w, sources):
    """dist and pred, one row per source.  float32 weights: distances in float64, no predecessors
    (they follow from float32 rounding)."""
    f32 = w.is_floating_point()
    w64 = w.double() if f32 else w.long()
    dist, pred = [], []
    for s in sources:
        d, inf = _bellman_ford(V, src, dst, w64, int(s))
        dist.append(d if f32 else torch.where(d < inf, d, -1))
        if not f32:
            pred.append(_tree(V, src, dst, w64, d, inf))
    return torch.stack(dist), None if f32 else torch.stack(pred)


def exact(case, seed):
    kind = case["kind"]
    gen = _gen(seed)
    if kind == "prune" or case.get("graph") == "grid":
        return None  # minutes in plain torch
    if kind == "batch":
        dist, pred = [], []
        for (V, src, dst, w), sources in _batch_inputs(case, gen, np.random.default_rng(seed)):
            _, s, t, wk, _ = _csr64(V, src, dst, w)
            f32 = wk.is_floating_point()
            wk = wk.double() if f32 else wk.long()
            S, inf = len(sources), float("inf") if f32 else 1 << 62
            d = torch.full((S, V), inf, dtype=wk.dtype, device="cuda")
            d[torch.arange(S, device="cuda"), torch.from_numpy(sources.astype(np.int64)).cuda()] = 0
            ts = t.expand(S, -1)
            while True:  # all sources of the graph at once
                ds = d[:, s]
                n = d.scatter_reduce(1, ts, torch.where(ds < inf, ds + wk, inf), "amin")
                if torch.equal(n, d):
                    break
                d = n
            dist.append((d if f32 else torch.where(d < inf, d, -1)).flatten())
            if not f32:
                ds = d[:, s]
                cand = torch.where((ds < inf) & (ds + wk == d[:, t]), s.expand(S, -1), V)
                p = torch.full((S, V), V, dtype=torch.int64, device="cuda").scatter_reduce(1, ts, cand, "amin")
                pred.append(torch.where(p < V, p, -1).flatten())
        dist = torch.cat(dist)
        return dict(dist=dist if dist.is_floating_point() else dist.int(), pred=torch.cat(pred).int() if pred else None)
    V, src, dst, w = _edges(case, gen)
    row_ptr, s, t, wk, eid = _csr64(V, src, dst, w)
    if kind == "build":
        return dict(row_ptr=row_ptr.int(), col=t.int(), w=wk, eid=eid.int())
    if kind == "compact":
        kept = torch.nonzero(_keep(case, wk.numel(), gen)).flatten()
        s, t = s[kept], t[kept]
        B = (V + case["P"] - 1) // case["P"]
        cut = s // B != t // B
        return dict(row_ptr=torch.searchsorted(s, torch.arange(V + 1, device="cuda")).int(), col=t.int(), w=wk[kept],
                    eid=kept.int(), bounds=(torch.arange(case["P"] + 1, device="cuda") * B).clamp(max=V).int(),
                    inter=torch.bincount(s[cut] // B, minlength=case["P"]))
    if kind == "layout":
        ids, slots = _layout64(V, case["P"], s, t)
        key, order = torch.sort(slots[s] * V + slots[t])
        return dict(row_ptr=torch.searchsorted(key, torch.arange(V + 1, device="cuda") * V).int(),
                    col=(key % V).int(), w=wk[order], eid=order.int(), ids=ids.int(), slots=slots.int())
    sources = _sources(case, V, src, dst, gen)
    if kind == "solve":
        dist, pred = _solve64(V, s, t, wk, sources.tolist())
        return dict(dist=dist if wk.is_floating_point() else dist.int(), pred=None if pred is None else pred.int())
    if kind == "update":
        if case["layout"]:  # the changed edges are drawn among the stored ones
            _, slots = _layout64(V, case["P"], s, t)
            order = torch.sort(slots[s] * V + slots[t]).indices
            s, t, wk = s[order], t[order], wk[order]
        dist, pred = _solve64(V, s, t, _changed(case, wk, gen)[1], sources.tolist())
        return dict(dist=dist if wk.is_floating_point() else dist.int(), pred=None if pred is None else pred.int())
    # grad: distances in float64; the gradient over the float32 shortest-path tree, summed in float64
    grad_dist = torch.randn((case["S"], V), generator=gen, device="cuda")
    dist = _solve64(V, s, t, wk, sources.tolist())[0]
    grad = torch.zeros(wk.numel(), dtype=torch.float64, device="cuda")
    key = s * V + t
    for i, x in enumerate(sources.tolist()):
        d, inf = _bellman_ford(V, s, t, wk, x)
        p = _tree(V, s, t, wk, d, inf)
        acc = grad_dist[i].double()
        hops = torch.where(p < 0, 0, -1)
        depth = 0
        while True:  # hop count of every vertex below the source
            nxt = (hops < 0) & (hops[p.clamp(min=0)] == depth)
            if not bool(nxt.any()):
                break
            depth += 1
            hops[nxt] = depth
        for h in range(depth, 0, -1):  # children before parents
            v = torch.nonzero(hops == h).flatten()
            grad.index_add_(0, torch.searchsorted(key, p[v] * V + v), acc[v])
            acc = acc.index_add(0, p[v], acc[v])
    return dict(dist=dist, grad_w=grad)
