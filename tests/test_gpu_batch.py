"""The batched solve in shared memory against the CPU oracle, at the sizes where its layouts change: up to
47,104 vertices (of all copies of a graph that a block solves together) and the general kernel past
them; one to 17 sources a graph; rows at the bounds of a hub (512 edges), more hub segments in a round
than their list holds; narrow and wide buckets, graphs of high diameter, no predecessors and bad edges.
Integer results and float32 distances are compared bit for bit."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def sssp():
    import paper_2103_12012_gb300 as m
    m.lib()
    return m


def u32(t):
    return t.detach().cpu().numpy().view(np.uint32)


def graph(rng, V, E, f32=False, hub=0):
    src, dst = rng.integers(0, V, E).astype(np.uint32), rng.integers(0, V, E).astype(np.uint32)
    if hub:
        src[:hub] = 3
        dst[:hub] = np.arange(hub) % V
    w = rng.uniform(0.5, 2.0, E).astype(np.float32) if f32 else rng.integers(1, 256, E).astype(np.uint32)
    return oracle.csr(V, src, dst, w)


def path(V, k, f32=False):
    """Edges from each vertex to the next k: a sweep takes about V / k iterations."""
    src = np.repeat(np.arange(V, dtype=np.uint32), k)
    dst = np.minimum(src + np.tile(np.arange(1, k + 1, dtype=np.uint32), V), V - 1).astype(np.uint32)
    keep = src != dst
    w = 1 + (src[keep] * 7 + dst[keep]) % 13
    return oracle.csr(V, src[keep], dst[keep], w.astype(np.float32 if f32 else np.uint32))


def check(b, graphs, preds=True, step=1):
    st, _ = b.status()
    assert st == 0
    for i in range(0, b.n_problems, step):
        gi, s = int(b.prob_graph[i]), int(b.prob_source[i])
        d, p, _ = oracle.dijkstra(graphs[gi], s)
        bd, bp = b.result(i)
        assert np.array_equal(u32(bd), d.view(np.uint32)), f"dist, problem {i}"
        if preds:
            assert np.array_equal(u32(bp), p), f"pred, problem {i}"


@pytest.mark.parametrize("f32", [False, True])
def test_sources_and_copies(sssp, f32):
    """Every count of sources from 1 to 17, with enough problems that blocks take several of them."""
    rng = np.random.default_rng(5 + f32)
    graphs, sources = [], []
    for S in range(1, 18):
        for V in (1, 2, 31, 33, 1000, 2944, 2945):
            graphs.append(graph(rng, V, 8 * V + 3, f32, hub=min(2500, 4 * V) if S % 3 == 0 and V > 3 else 0))
            sources.append(rng.integers(0, V, S).tolist())
    for V in (64, 100, 6000):  # (thousands of problems: up to 16 copies a block)
        graphs.append(graph(rng, V, 6 * V, f32))
        sources.append(rng.integers(0, V, 3001 if V < 6000 else 17).tolist())
    b = sssp.Batch(graphs, sources, sssp.options(delta=0.16 if f32 else 16.0))
    b.solve()
    check(b, graphs)
    b.dist.fill_(0)
    b.pred.fill_(0)
    b.make_plan()
    for _ in range(2):
        b.replay()
    check(b, graphs)


@pytest.mark.parametrize("delta", [1.0, 16.0, 1e9])
@pytest.mark.parametrize("f32", [False, True])
def test_graph_sizes(sssp, f32, delta):
    rng = np.random.default_rng(3)
    if f32:
        delta /= 100.0
    for sizes in ((8191, 8192), (8193, 16000), (47103, 47104), (1000, 47105, 65537)):
        graphs = [graph(rng, V, 3 * V, f32, hub=V // 2) for V in sizes]
        sources = [[3, g.V - 1] for g in graphs]
        b = sssp.Batch(graphs, sources, sssp.options(delta=delta, threads=1024, tile=2048))
        b.solve()
        check(b, graphs)


def test_large_and_small_ends_together(sssp):
    """More large problems than blocks: the order of processing takes from both ends."""
    rng = np.random.default_rng(8)
    graphs = [graph(rng, V, 2 * V) for V in (47200, 300, 48000, 20000)]
    sources = [rng.integers(0, g.V, n).tolist() for g, n in zip(graphs, (200, 60, 150, 20))]
    b = sssp.Batch(graphs, sources, sssp.options(delta=32.0))
    b.make_plan()
    b.replay()
    check(b, graphs, step=9)


def test_large_batch_split_over_both_kernels(sssp):
    """Large problems for several rounds of blocks, and small graphs among them."""
    rng = np.random.default_rng(12)
    graphs = [graph(rng, V, 2 * V) for V in (47200, 300, 47104)]
    sources = [rng.integers(0, g.V, n).tolist() for g, n in zip(graphs, (1300, 70, 9))]
    b = sssp.Batch(graphs, sources, sssp.options(delta=32.0))
    b.make_plan()
    for _ in range(2):
        b.replay()
    check(b, graphs, step=23)
    assert b.status()[1]["vertices"] > 0


@pytest.mark.parametrize("V", [38000, 47000])
def test_hub_rows(sssp, V):
    """Rows of 511, 512 and 513 edges, and three rows of every vertex in one round: more segments than
    their list holds."""
    rng = np.random.default_rng(V)
    src, dst = [np.full(3, 5)], [np.array([1, 2, 3])]
    for h in (1, 2, 3):
        src.append(np.full(V, h))
        dst.append(np.arange(V))
    for k, d in enumerate((31, 511, 512, 513, 1025)):
        for v in range(10 + 7 * k, V, 997):
            src.append(np.full(d, v))
            dst.append(rng.choice(V, d, replace=False))
    src, dst = np.concatenate(src).astype(np.uint32), np.concatenate(dst).astype(np.uint32)
    g = oracle.csr(V, src, dst, rng.integers(1, 50, src.size).astype(np.uint32))
    b = sssp.Batch([g], [[5, 10]], sssp.options(delta=64.0))
    b.solve()
    check(b, [g])


@pytest.mark.parametrize("f32", [False, True])
def test_paths(sssp, f32):
    graphs = [path(3000, 5, f32), path(45000, 40, f32), path(700, 1, f32)]
    sources = [[0, 1, 2, 3], [0, 5], [0] * 9]
    b = sssp.Batch(graphs, sources, sssp.options(delta=4.0))
    b.solve()
    check(b, graphs)


@pytest.mark.parametrize("S", [1, 3])
def test_without_predecessors(sssp, S):
    rng = np.random.default_rng(S)
    graphs = [graph(rng, V, 9 * V) for V in (500, 3001, 40000)]
    b = sssp.Batch(graphs, [rng.integers(0, g.V, S).tolist() for g in graphs], sssp.options(delta=16.0))
    b.c.pred = None
    b.solve()
    check(b, graphs, preds=False)


@pytest.mark.parametrize("V", [3000, 40000])
@pytest.mark.parametrize("what", ["head", "weight", "overflow"])
def test_bad_edges_are_reported(sssp, V, what):
    rng = np.random.default_rng(1)
    g = graph(rng, V, 10 * V)
    e = int(g.row_ptr[17])
    if what == "head":
        g.col[e] = V
    else:
        g.w[e] = 0 if what == "weight" else 0xFFFFFFF0
    b = sssp.Batch([g], [[17, int(rng.integers(100, V)), 5]], sssp.options(delta=16.0))
    b.solve()
    assert b.status()[0] == (sssp.SSSP_EOVERFLOW if what == "overflow" else sssp.SSSP_EINVAL)


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("preds", [False, True])
@pytest.mark.parametrize("V", [2000, 40000])
def test_overflow_is_of_final_distances(sssp, V, preds, f32):
    """1 is lowered within a bucket, after it has been relaxed; its candidate for 3 fits only then, or not at
    all."""
    rng = np.random.default_rng(V)
    dt, unit, way, fits, not_fits = (np.float32, 1e38, 2.9, 1, 3) if f32 else (np.uint32, 1000000000, 2, 2.5, 4)
    src, dst = rng.integers(10, V, (2, 4 * V)).astype(np.uint32)
    w = rng.integers(1, 256, src.size)
    for last in (fits, not_fits):
        extra = [(0, 1, way), (0, 2, 0.5), (2, 1, 0.5), (1, 3, last), (0, 10, 1 / unit)]
        g = oracle.csr(V, np.append(src, [a for a, _, _ in extra]).astype(np.uint32),
                       np.append(dst, [b for _, b, _ in extra]).astype(np.uint32),
                       np.append(w, [c * unit for _, _, c in extra]).astype(dt))
        b = sssp.Batch([g], [[0, 10]], sssp.options(delta=unit))
        if not preds:
            b.c.pred = None
        b.solve()
        assert b.status()[0] == (0 if last == fits else sssp.SSSP_EOVERFLOW)
        for i in range(2):
            d, p, _ = oracle.dijkstra(g, 10 * i)
            bd, bp = b.result(i)
            assert np.array_equal(u32(bd), d.view(np.uint32)) and (not preds or np.array_equal(u32(bp), p))


@pytest.mark.parametrize("V", [40, 3000, 20000])
def test_sources_that_reach_little(sssp, V):
    """Isolated sources, sources with a few edges or a long row into vertices without edges, and sources that
    reach an eighth of the graph and more, as copies of one graph."""
    rng = np.random.default_rng(V)
    k = V // 8
    src, dst = rng.integers(k, V, 6 * V), rng.integers(k, V, 6 * V)  # vertices from k on; the first ones are apart
    few = np.stack([[1, 1, 2, 3], [2, 3, 4, 4]])
    row = np.stack([np.full(k - 5, 4), np.arange(5, k)]) if V > 40 else np.zeros((2, 0), int)
    half = np.stack([np.arange(k, k + V // 16), np.arange(k + 1, k + 1 + V // 16)])
    src, dst = np.concatenate([src, few[0], row[0], half[0]]), np.concatenate([dst, few[1], row[1], half[1]])
    g = oracle.csr(V, src.astype(np.uint32), dst.astype(np.uint32), rng.integers(1, 9, src.size).astype(np.uint32))
    sources = [0, 1, 2, 4, V - 1, k, 0, 3, V - 2, 1, 0, 4]
    graphs = [g] + [graph(rng, 300, 1500) for _ in range(3)]
    b = sssp.Batch(graphs, [sources, [1], [2] * 17, [5]], sssp.options(delta=3.0))
    for _ in range(2):
        b.solve()
        check(b, graphs)


@pytest.mark.parametrize("kind", ["dense", "very dense", "grids"])
@pytest.mark.parametrize("delta", [0.0, 40.0])
def test_graphs_that_shared_memory_leaves(sssp, kind, delta):
    """Dense graphs and grids, with few and with many problems, at the default and a given width; a workspace of the
    size for other options does."""
    rng = np.random.default_rng(len(kind))
    if kind == "grids":
        at = np.arange(100 * 90).reshape(100, 90)
        a, c = np.concatenate([at[1:].ravel(), at[:, 1:].ravel()]), np.concatenate([at[:-1].ravel(), at[:, :-1].ravel()])
        g = oracle.csr(9000, np.concatenate([a, c]).astype(np.uint32), np.concatenate([c, a]).astype(np.uint32),
                       rng.integers(1, 99, 2 * a.size).astype(np.uint32))
    else:
        g = graph(rng, 600, 600 * (40 if kind == "dense" else 90))
    for n in (3, 1300):
        b = sssp.Batch([g], [rng.integers(0, g.V, n).tolist()], sssp.options())
        b.opts.delta = delta
        b.solve()
        check(b, [g], step=max(n // 9, 1))


@pytest.mark.parametrize("V,S", [(900, 3), (16000, 5)])
def test_rows_at_the_bound_of_segments(sssp, V, S):
    """Rows of 127, 128, 129, 255, 256 and 257 edges, relaxed in the same rounds as short ones."""
    rng = np.random.default_rng(V)
    src, dst = [rng.integers(0, V, 4 * V)], [rng.integers(0, V, 4 * V)]
    for k, d in enumerate((127, 128, 129, 255, 256, 257)):
        for v in range(k, V, 100):
            src.append(np.full(d, v))
            dst.append(rng.choice(V, d, replace=False))
    src, dst = np.concatenate(src).astype(np.uint32), np.concatenate(dst).astype(np.uint32)
    g = oracle.csr(V, src, dst, rng.integers(1, 200, src.size).astype(np.uint32))
    b = sssp.Batch([g] * 70, [rng.integers(0, V, S).tolist() for _ in range(70)], sssp.options(delta=16.0))
    b.solve()
    check(b, [g] * 70, step=7)


@pytest.mark.parametrize("V", [3000, 40000])
def test_limit_ends_a_batch(sssp, V):
    """A limit of a nanosecond ends the batch with a status; the next call in the same workspace is right."""
    rng = np.random.default_rng(V)
    g = graph(rng, V, 8 * V)
    b = sssp.Batch([g], [rng.integers(0, V, 400).tolist()], sssp.options(delta=16.0, timeout_ns=1))
    b.solve()
    assert b.status()[0] == sssp.SSSP_ETIMEOUT
    b.opts.timeout_ns = 0
    b.solve()
    check(b, [g], step=40)
