"""The sweep (sssp_solve on graphs of five edges per vertex and more in the default policy) against
the CPU oracle, at the sizes where its layouts change: one to 33 sources (rows of 1, 2, 4 and 8
distances, several groups, padded lanes), rows around the list bounds (31/32, 511/512/513 edges and
hubs of several segments), ids and distances at the edges of their ranges, and the hand-over to the
persistent solve.  Integer results and float32 distances are compared bit for bit."""
import ctypes

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


def check(sssp, g, ref, sources, opts=None, status=0):
    dist, pred, st, stats = sssp.solve(g, np.asarray(sources, np.uint32), opts, check=False)
    assert st == status
    for i, s in enumerate(sources):
        d, p, _ = oracle.dijkstra(ref, int(s))
        assert np.array_equal(u32(dist[i]), d.view(np.uint32)), f"dist, source {s}"
        assert np.array_equal(u32(pred[i]), p), f"pred, source {s}"
    return stats


def graph(rng, V, E, f32=False, hi=255):
    src, dst = rng.integers(0, V, E).astype(np.uint32), rng.integers(0, V, E).astype(np.uint32)
    w = rng.uniform(0.5, 2.0, E).astype(np.float32) if f32 else rng.integers(1, hi + 1, E).astype(np.uint32)
    return src, dst, w


@pytest.mark.parametrize("S", [1, 2, 3, 4, 5, 8, 9, 17, 33])
@pytest.mark.parametrize("V", [64, 65, 2049, 20011])
@pytest.mark.parametrize("f32", [False, True])
def test_sources_and_sizes(sssp, S, V, f32):
    rng = np.random.default_rng(1000 * S + V)
    src, dst, w = graph(rng, V, 9 * V + 5, f32)
    ref = oracle.csr(V, src, dst, w)
    g = sssp.build_csr(V, src, dst, w)
    check(sssp, g, ref, rng.integers(0, V, S).tolist())


@pytest.mark.parametrize("layout", [False, True])
@pytest.mark.parametrize("S", [1, 4, 12])
def test_rows_at_the_list_bounds_and_hubs(sssp, layout, S):
    """Rows of 0, 1, 31, 32, 33, 511, 512, 513 and several thousand edges, many of each marked in one
    iteration (every vertex is reached from a hub)."""
    rng = np.random.default_rng(7 + S)
    V = 9000
    degs = np.array([0, 1, 31, 32, 33, 127, 128, 511, 512, 513, 1025, 4000])
    tails, heads = [], []
    for v in range(0, V, 3):
        d = int(degs[(v // 3) % len(degs)]) if v else V - 1
        if d > 600 and v > 300:
            d = 33
        h = rng.choice(V, d, replace=False)
        tails.append(np.full(h.size, v))
        heads.append(h)
    src, dst = np.concatenate(tails).astype(np.uint32), np.concatenate(heads).astype(np.uint32)
    w = rng.integers(1, 1000, src.size).astype(np.uint32)
    ref = oracle.csr(V, src, dst, w)
    g = sssp.build_csr(V, src, dst, w, partitions=5)
    if layout:
        g = sssp.layout(g)
    check(sssp, g, ref, [0, 3, 6, 300, 1, 8997, 0, 9, 12, 15, 18, 21][:S])


def test_power_law_graph_with_layout_and_unreached_part(sssp):
    g0 = gg.rmat(gg.BASE_SEED + 700, 15, 16 << 15)
    ref = oracle.csr_of(g0)
    h = sssp.layout(sssp.build_csr(g0.V, g0.src, g0.dst, g0.w, partitions=37))
    srcs = gg.pick_sources(gg.BASE_SEED + 700, g0, 10).tolist()
    stats = check(sssp, h, ref, srcs, sssp.options(delta=10, hub_count=64))
    assert stats["rounds"] < 200 and stats["remote_activations"] == 0  # (swept: no units, no messages)


@pytest.mark.parametrize("S", [1, 3, 8, 10])
@pytest.mark.parametrize("f32", [False, True])
def test_hand_over_on_a_high_diameter_graph(sssp, S, f32):
    """A band graph (vertex v to v+1 .. v+7 and back) has 14 edges per vertex and thousands of hops:
    the sweep gives up and the persistent solve finishes from its state."""
    rng = np.random.default_rng(5)
    V = 30000
    v = np.repeat(np.arange(V), 7)
    t = v + np.tile(np.arange(1, 8), V)
    keep = t < V
    src = np.concatenate([v[keep], t[keep]]).astype(np.uint32)
    dst = np.concatenate([t[keep], v[keep]]).astype(np.uint32)
    w = rng.uniform(0.5, 2.0, src.size).astype(np.float32) if f32 else rng.integers(1, 50, src.size).astype(np.uint32)
    ref = oracle.csr(V, src, dst, w)
    g = sssp.build_csr(V, src, dst, w, partitions=3)
    stats = check(sssp, g, ref, [0, V - 1, V // 2, 7, 77, 777, 7777, 17777, 1, 2][:S])
    assert stats["remote_activations"] > 0  # messages between the persistent solve's units


def test_overflow_bad_source_bad_edge(sssp):
    V = 500
    rng = np.random.default_rng(9)
    src, dst, w = graph(rng, V, 5000)
    w[::50] = 0xFFFFFFF0  # sums beyond uint32 on some paths
    ref = oracle.csr(V, src, dst, w)
    g = sssp.build_csr(V, src, dst, w)
    check(sssp, g, ref, [0, 1], status=sssp.SSSP_EOVERFLOW)
    dist, _, st, _ = sssp.solve(g, np.array([3, V, 4], np.uint32), check=False)
    assert st == sssp.SSSP_EINVAL and (u32(dist[1]) == 0xFFFFFFFF).all()
    clean = graph(rng, V, 5000)
    ref = oracle.csr(V, *clean)
    col = ref.col.copy()
    col[int(ref.row_ptr[5])] = V + 9  # a head that is no vertex: reported, not followed
    _, _, st, _ = sssp.solve(sssp.upload_csr(V, ref.row_ptr, col, ref.w), np.array([5], np.uint32), check=False)
    assert st == sssp.SSSP_EINVAL


def test_without_predecessors_and_in_an_unaligned_workspace(sssp):
    """pred NULL, and a workspace that is aligned to 16 bytes only (rows of eight need 32)."""
    V, S = 4001, 6
    rng = np.random.default_rng(11)
    src, dst, w = graph(rng, V, 8 * V)
    ref = oracle.csr(V, src, dst, w)
    g = sssp.build_csr(V, src, dst, w)
    gc, o = g.c(), sssp.options()
    sources = torch.arange(S, dtype=torch.int32, device="cuda") * 600
    need = sssp.lib().sssp_solve_workspace_size(ctypes.byref(gc), S, ctypes.byref(o))
    for off in (0, 16):
        ws = torch.empty(need + 64, dtype=torch.uint8, device="cuda")
        p = ws.data_ptr() + (-ws.data_ptr()) % 32 + off
        dist = torch.empty((S, V), dtype=torch.int32, device="cuda")
        pred = torch.empty((S, V), dtype=torch.int32, device="cuda")
        for q in (None, ctypes.c_void_p(pred.data_ptr())):
            dist.fill_(7)
            assert sssp.lib().sssp_solve(ctypes.byref(gc), ctypes.c_void_p(sources.data_ptr()), S,
                                         ctypes.c_void_p(dist.data_ptr()), q, ctypes.byref(o), ctypes.c_void_p(p),
                                         need, sssp._stream()) == sssp.SSSP_OK
            assert sssp.lib().sssp_workspace_status(ctypes.c_void_p(p), sssp._stream(), None) == sssp.SSSP_OK
            for i in range(S):
                d, pr, _ = oracle.dijkstra(ref, 600 * i)
                assert np.array_equal(u32(dist[i]), d)
                assert q is None or np.array_equal(u32(pred[i]), pr)


@pytest.mark.parametrize("S", [1, 2, 3, 4, 6, 8, 12])
@pytest.mark.parametrize("layout", [False, True])
@pytest.mark.parametrize("f32", [False, True])
def test_warm_start(sssp, S, layout, f32):
    """Many tails (some listed twice): rows of 1, 2 and 4 packed words, several groups, hubs among the
    tails, ties that a lower label wins."""
    rng = np.random.default_rng(10 * S + layout)
    V, E = 30011, 260000
    src, dst, w = graph(rng, V, E, f32, hi=9)
    src[:3000], dst[:3000] = 7, np.arange(3000)
    src[3000:9000], dst[3000:9000] = 11, np.arange(6000)
    sources = rng.integers(0, V, S).astype(np.uint32)
    sources[0] = 7
    g = sssp.build_csr(V, src, dst, w, partitions=13)
    dist, pred = sssp.solve(sssp.layout(g) if layout else g, sources)[:2]
    at = rng.permutation(E)[:17000]
    w2 = w.copy()
    w2[at] = w[at] * np.float32(0.6) if f32 else np.maximum(1, w[at] // 2)
    g2 = sssp.build_csr(V, src, dst, w2, partitions=13)
    dist, pred, st, stats = sssp.update(sssp.layout(g2) if layout else g2, dist, pred,
                                        np.concatenate([src[at], src[at[:100]]]))
    assert st == 0
    ref = oracle.csr(V, src, dst, w2)
    for i, s in enumerate(sources):
        d, p, _ = oracle.dijkstra(ref, int(s))
        assert np.array_equal(u32(dist[i]), d.view(np.uint32)), f"dist, source {s}"
        assert np.array_equal(u32(pred[i]), p), f"pred, source {s}"


@pytest.mark.parametrize("S", [1, 4])
@pytest.mark.parametrize("kind", ["full lists", "chain"])
def test_warm_start_handed_over(sssp, S, kind):
    """More items than a list holds, and a chain of more iterations than a warm sweep takes."""
    rng = np.random.default_rng(S)
    if kind == "full lists":
        V = 40000
        src, dst, w = graph(rng, V, 6 * V)
        w2 = np.maximum(1, w // 3).astype(np.uint32)
        tails = src
    else:  # each vertex to the next six
        V = 20000
        src = np.repeat(np.arange(V - 6), 6).astype(np.uint32)
        dst = src + np.tile(np.arange(1, 7), V - 6).astype(np.uint32)
        w = rng.integers(50, 60, src.size).astype(np.uint32)
        w2 = w.copy()
        w2[:12] = 1
        tails = np.concatenate([src[:12], np.full(20000, V - 1, np.uint32)])
    sources = np.arange(S).astype(np.uint32)
    dist, pred = sssp.solve(sssp.build_csr(V, src, dst, w), sources)[:2]
    dist, pred, st, _ = sssp.update(sssp.build_csr(V, src, dst, w2), dist, pred, tails)
    assert st == 0
    ref = oracle.csr(V, src, dst, w2)
    for i, s in enumerate(sources):
        d, p, _ = oracle.dijkstra(ref, int(s))
        assert np.array_equal(u32(dist[i]), d), f"dist, source {s}"
        assert np.array_equal(u32(pred[i]), p), f"pred, source {s}"


def test_warm_start_with_a_bad_tail(sssp):
    rng = np.random.default_rng(4)
    V = 20000
    src, dst, w = graph(rng, V, 8 * V)
    g = sssp.build_csr(V, src, dst, w)
    dist, pred = sssp.solve(g, np.array([3, 4], np.uint32))[:2]
    d0, p0 = dist.clone(), pred.clone()
    tails = src.copy()
    tails[5] = V
    dist, pred, st, _ = sssp.update(g, dist, pred, tails, check=False)
    assert st == sssp.SSSP_EINVAL
    assert torch.equal(dist, d0) and torch.equal(pred, p0)


@pytest.mark.parametrize("S", [1, 2, 4, 8, 9])
@pytest.mark.parametrize("f32", [False, True])
def test_marks_under_contention(sssp, S, f32):
    """A small dense graph: every iteration lowers most distances several times from many warps while their
    items are taken, so an item whose mark is set and cleared in the wrong order keeps a distance that
    is too large.  Repeated, with the same result each time."""
    rng = np.random.default_rng(70 + S)
    V = 3001
    src, dst, w = graph(rng, V, 150 * V, f32, hi=1000000)
    ref = oracle.csr(V, src, dst, w)
    g = sssp.build_csr(V, src, dst, w, partitions=5)
    sources = rng.integers(0, V, S).astype(np.uint32)
    stats = check(sssp, g, ref, sources.tolist())
    assert stats["remote_activations"] == 0 and stats["rounds"] > 0  # (swept)
    first = [t.clone() for t in sssp.solve(g, sources)[:2]]
    solver = sssp.Solver(g, S)
    for _ in range(50):
        dist, pred = solver(sources)
        assert torch.equal(dist, first[0]) and torch.equal(pred, first[1])


@pytest.mark.parametrize("S", [1, 2, 3, 4, 8])
def test_warm_ties_under_contention(sssp, S):
    """Weights 1 and 2: most vertices have many predecessors of one distance, whose labels several warps lower
    while others read the packed words; the least label wins each time."""
    rng = np.random.default_rng(80 + S)
    V, E = 60011, 20 * 60011
    src, dst, w = graph(rng, V, E, hi=2)
    w0 = w + np.where((src < 9000) & (rng.random(E) < 0.05), 2, 0).astype(np.uint32)
    ref = oracle.csr(V, src, dst, w)
    g = sssp.build_csr(V, src, dst, w, partitions=5)
    sources = rng.integers(0, V, S).astype(np.uint32)
    want = [oracle.dijkstra(ref, int(s)) for s in sources]
    dist0, pred0 = sssp.solve(sssp.build_csr(V, src, dst, w0, partitions=5), sources)[:2]
    for _ in range(10):
        dist, pred, st, stats = sssp.update(g, dist0.clone(), pred0.clone(), np.arange(17000, dtype=np.uint32))
        assert st == 0 and stats["remote_activations"] == 0  # (swept)
        for i, (d, p, _) in enumerate(want):
            assert np.array_equal(u32(dist[i]), d) and np.array_equal(u32(pred[i]), p)
