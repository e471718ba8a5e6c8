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


def fits(ref, sources):
    """Every candidate from a final distance can be represented (else the status is SSSP_EOVERFLOW)."""
    tail = np.repeat(np.arange(ref.row_ptr.size - 1), np.diff(ref.row_ptr.astype(np.int64)))
    for s in sources:
        d = oracle.dijkstra(ref, int(s))[0]
        if ref.w.dtype == np.float32:
            d, w = d.view(np.float32), ref.w
            on = np.isfinite(d[tail])
            with np.errstate(over="ignore"):
                c, top = d[tail][on] + w[on], np.float32(np.inf)
        else:
            on = d[tail] != 0xFFFFFFFF
            c, top = d[tail][on].astype(np.uint64) + ref.w[on], 0xFFFFFFFF
        if (c >= top).any():
            return False
    return True


@pytest.mark.parametrize("S", [1, 2, 4, 9])
@pytest.mark.parametrize("f32", [False, True])
def test_overflow_is_of_final_distances(sssp, S, f32):
    """Weights up to a quarter of the range: distances on the way are past its end, final ones not; then one
    edge from a reached vertex whose final candidate is."""
    rng = np.random.default_rng(90 + S)
    V = 16384
    src, dst, w = graph(rng, V, 8 * V, hi=(1 << 30) - 1)
    if f32:
        w = (w * 8e28).astype(np.float32)
    sources = rng.integers(0, V, S)
    ref = oracle.csr(V, src, dst, w)
    assert fits(ref, sources)
    stats = check(sssp, sssp.build_csr(V, src, dst, w, partitions=5), ref, sources.tolist())
    assert stats["remote_activations"] == 0  # (swept)
    u = int(oracle.dijkstra(ref, int(sources[0]))[0].view(np.float32 if f32 else np.uint32).argsort()[V // 2])
    w[np.nonzero(src == u)[0][0]] = np.float32(3.4e38) if f32 else 0xFFFFFFFE
    ref = oracle.csr(V, src, dst, w)
    assert not fits(ref, sources)
    check(sssp, sssp.build_csr(V, src, dst, w, partitions=5), ref, sources.tolist(), status=sssp.SSSP_EOVERFLOW)


@pytest.mark.parametrize("S", [1, 3, 8])
@pytest.mark.parametrize("final", [False, True])
def test_overflow_when_handed_over(sssp, S, final):
    """A band graph, which the persistent solve finishes.  A long cut makes candidates on the way that do not
    fit; or a vertex that the sweep is done with has one."""
    rng = np.random.default_rng(6)
    V = 30000
    v = np.repeat(np.arange(V), 7)
    t = v + np.tile(np.arange(1, 8), V)
    keep = t < V
    src = np.concatenate([v[keep], t[keep], [0]]).astype(np.uint32)
    dst = np.concatenate([t[keep], v[keep], [15000]]).astype(np.uint32)
    w = rng.integers(1, 50, src.size).astype(np.uint32)
    w[-1] = 3000000000
    w[(src == 15000) & (dst == 15001)] = 2000000000
    if final:
        w[(src == 12) & (dst == 13)] = 0xFFFFFFFE
    sources = [0, 3, 1, 2, 4, 5, 6, 7][:S]
    ref = oracle.csr(V, src, dst, w)
    assert fits(ref, sources) == (not final)
    check(sssp, sssp.build_csr(V, src, dst, w), ref, sources, status=sssp.SSSP_EOVERFLOW if final else 0)


@pytest.mark.parametrize("S", [1, 2, 4])
@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("kind", ["on the way", "final", "not touched"])
def test_overflow_in_a_warm_start(sssp, S, f32, kind):
    """The changed edges' heads get distances that a shorter way replaces; one vertex that is reached anew has
    a candidate that does not fit; or one that the change does not reach."""
    rng = np.random.default_rng(95 + S)
    V = 60011
    dt, unit = (np.float32, 1e38) if f32 else (np.uint32, 1200000000)  # (3 units fit, 4 do not)
    src, dst, w = graph(rng, V, 8 * V, f32)
    keep = (dst >= 10) & (src >= 10)
    extra = [(0, 1, 3), (0, 2, 1), (2, 1, 1), (1, 3, 3 if kind == "final" else 1), (0, 20, 1 / unit), (0, 6, 2)]
    if kind == "not touched":
        extra.append((6, 9, 3))
    src = np.concatenate([src[keep], [a for a, _, _ in extra]]).astype(np.uint32)
    dst = np.concatenate([dst[keep], [b for _, b, _ in extra]]).astype(np.uint32)
    w = np.concatenate([w[keep], [c * unit for _, _, c in extra]]).astype(dt)
    before = ~((src == 0) & (dst < 3))  # the edges 0 -> 1 and 0 -> 2 are added
    sources = np.zeros(S, np.uint32)
    dist, pred = sssp.solve(sssp.build_csr(V, src[before], dst[before], w[before], partitions=5), sources, check=False)[:2]
    ref = oracle.csr(V, src, dst, w)
    assert fits(ref, sources) == (kind == "on the way")
    dist, pred, st, stats = sssp.update(sssp.build_csr(V, src, dst, w, partitions=5), dist, pred,
                                        np.zeros(17000, np.uint32), check=False)
    assert stats["remote_activations"] == 0  # (swept)
    assert st == (sssp.SSSP_EOVERFLOW if kind == "final" else 0)
    d, p, _ = oracle.dijkstra(ref, 0)
    for i in range(S):
        assert np.array_equal(u32(dist[i]), d.view(np.uint32)) and np.array_equal(u32(pred[i]), p)


@pytest.mark.parametrize("S", [1, 4])
def test_overflow_in_a_warm_start_that_is_handed_over(sssp, S):
    """An item of the first iterations has a candidate that does not fit; the persistent solve finishes."""
    rng = np.random.default_rng(S)
    V = 20000
    src = np.repeat(np.arange(V - 6), 6).astype(np.uint32)
    dst = src + np.tile(np.arange(1, 7), V - 6).astype(np.uint32)
    w = rng.integers(50, 60, src.size).astype(np.uint32)
    src, dst, w = np.append(src, 9).astype(np.uint32), np.append(dst, 900).astype(np.uint32), np.append(w, np.uint32(0xFFFFFFFE))
    w2 = w.copy()
    w2[:12] = 1
    sources = np.arange(S).astype(np.uint32)
    dist, pred = sssp.solve(sssp.build_csr(V, src, dst, w), sources, check=False)[:2]
    dist, pred, st, _ = sssp.update(sssp.build_csr(V, src, dst, w2), dist, pred,
                                    np.concatenate([src[:12], np.full(20000, V - 1, np.uint32)]), check=False)
    assert st == sssp.SSSP_EOVERFLOW
    ref = oracle.csr(V, src, dst, w2)
    for i, s in enumerate(sources):
        d, p, _ = oracle.dijkstra(ref, int(s))
        assert np.array_equal(u32(dist[i]), d) and np.array_equal(u32(pred[i]), p)


@pytest.mark.parametrize("S", [1, 3, 8])
@pytest.mark.parametrize("f32", [False, True])
def test_tail_is_handed_over(sssp, S, f32):
    """A random graph, which the sweep is done with in some iterations, with a path of thousands of hops behind
    it, which the persistent solve follows from what the sweep leaves."""
    rng = np.random.default_rng(3)
    V, n = 30000, 6000
    src, dst, w = graph(rng, V, 9 * V, f32)
    src = np.concatenate([src, [7], np.arange(V, V + n - 1)]).astype(np.uint32)
    dst = np.concatenate([dst, np.arange(V, V + n)]).astype(np.uint32)
    w = np.concatenate([w, np.full(n, 3, w.dtype)])
    ref = oracle.csr(V + n, src, dst, w)
    g = sssp.build_csr(V + n, src, dst, w, partitions=19)
    stats = check(sssp, g, ref, rng.integers(0, V, S).tolist())
    assert stats["remote_activations"] > 0  # messages between the persistent solve's units


@pytest.mark.parametrize("S,delta", [(1, 0.0), (1, 48.0), (3, 0.0), (3, 48.0), (8, 0.0)])
@pytest.mark.parametrize("kind", ["u32", "f32", "units"])
def test_graphs_of_many_hops(sssp, S, delta, kind):
    """A lattice: after the first iterations the persistent solve takes over from the sources, or the sweep
    goes on (few units and buckets far below the weights)."""
    rng = np.random.default_rng(4)
    n = 24
    at = np.arange(n ** 3).reshape(n, n, n)
    pairs = [(at[1:].ravel(), at[:-1].ravel()), (at[:, 1:].ravel(), at[:, :-1].ravel()),
             (at[:, :, 1:].ravel(), at[:, :, :-1].ravel())]
    src = np.concatenate([a for a, _ in pairs] + [b for _, b in pairs]).astype(np.uint32)
    dst = np.concatenate([b for _, b in pairs] + [a for a, _ in pairs]).astype(np.uint32)
    if kind == "f32":
        w, delta = rng.uniform(0.5, 2.0, src.size).astype(np.float32), delta / 100
    else:
        w = rng.integers(1, 256 if kind == "u32" else 2, src.size).astype(np.uint32)
    ref = oracle.csr(n ** 3, src, dst, w)
    stats = check(sssp, sssp.build_csr(n ** 3, src, dst, w, partitions=7), ref, rng.integers(0, n ** 3, S).tolist(),
                  sssp.options(delta=delta))
    kept = delta == 0.0 and kind != "units"
    assert (stats["remote_activations"] == 0) == kept


@pytest.mark.parametrize("S", [1, 4, 9])
def test_limit_of_a_sweep_ends_it(sssp, S):
    """A limit of a nanosecond ends the waits of a cold and of a warm sweep with a status; the hand-over behind them
    passes, and the next call in the same workspace is right."""
    rng = np.random.default_rng(S)
    V = 60000
    src, dst, w = graph(rng, V, 8 * V)
    w2 = np.maximum(1, w // 2).astype(np.uint32)
    g, g2 = sssp.build_csr(V, src, dst, w, partitions=9), sssp.build_csr(V, src, dst, w2, partitions=9)
    sources = torch.from_numpy(rng.integers(0, V, S).astype(np.int32)).cuda()
    tails = torch.arange(17000, dtype=torch.int32, device="cuda")
    cold, warm = sssp.Solver(g, S, sssp.options(timeout_ns=1)), sssp.Solver(g2, S, sssp.options(timeout_ns=1))
    cold(sources, check=False)
    assert cold.last_status == sssp.SSSP_ETIMEOUT
    cold.opts.timeout_ns = 0
    dist, pred = cold(sources)
    assert cold.last_stats["remote_activations"] == 0  # (swept)
    for i, s in enumerate(sources.tolist()):
        d, p, _ = oracle.dijkstra(oracle.csr(V, src, dst, w), s)
        assert np.array_equal(u32(dist[i]), d) and np.array_equal(u32(pred[i]), p)
    warm.update(dist.clone(), pred.clone(), tails)
    assert warm.status()[0] == sssp.SSSP_ETIMEOUT
    warm.opts.timeout_ns = 0
    dist, pred = warm.update(dist.clone(), pred.clone(), torch.arange(V, dtype=torch.int32, device="cuda"))
    assert warm.status()[0] == 0
    for i, s in enumerate(sources.tolist()):
        d, p, _ = oracle.dijkstra(oracle.csr(V, src, dst, w2), s)
        assert np.array_equal(u32(dist[i]), d) and np.array_equal(u32(pred[i]), p)


def test_two_streams_and_few_blocks(sssp):
    """Sweeps on two streams at a time, one of them with one block per SM."""
    rng = np.random.default_rng(2)
    V, S = 50000, 6
    src, dst, w = graph(rng, V, 8 * V)
    ref = oracle.csr(V, src, dst, w)
    g = sssp.build_csr(V, src, dst, w)
    streams = [torch.cuda.Stream() for _ in range(2)]
    solvers = [sssp.Solver(g, S), sssp.Solver(g, S, sssp.options(blocks_per_sm=1))]
    sources = [torch.from_numpy(rng.integers(0, V, S).astype(np.int32)).cuda() for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(10):
        for k in range(2):
            solvers[k].launch(sources[k], stream=streams[k])
    for k in range(2):
        assert solvers[k].status(streams[k])[0] == 0
        for i, s in enumerate(sources[k].tolist()):
            d, p, _ = oracle.dijkstra(ref, s)
            assert np.array_equal(u32(solvers[k].dist[i]), d) and np.array_equal(u32(solvers[k].pred[i]), p)
