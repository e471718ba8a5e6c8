"""The one-time graph steps at the sizes where their kernels change path: partition counts up to a
vertex each (ranges that cross many partitions, empty ones among them), compaction around its mask
words and tiles and with an unaligned keep mask, the prune around its blocks and shares, all against the CPU oracle (integers: equal)."""
import numpy as np
import pytest

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


def edges(seed, V, E, hi=255):
    rng = np.random.default_rng(seed)
    return (rng.integers(0, V, E).astype(np.uint32), rng.integers(0, V, E).astype(np.uint32),
            rng.integers(1, hi + 1, E).astype(np.uint32))


@pytest.mark.parametrize("V,E,P", [(1, 3, 1), (40, 0, 7), (300, 90000, 300), (70000, 200000, 70000),
                                   (70000, 200000, 3), (5000, 4095, 33), (100001, 1200000, 148)])
def test_partition_counts(sssp, V, E, P):
    src, dst, w = edges(V + P, V, E)
    src[: E // 2] %= max(V // 3, 1)  # a tail of vertices without edges, a heavy part
    ref = oracle.csr(V, src, dst, w)
    g = sssp.build_csr(V, src, dst, w, partitions=P)
    b, inter = sssp.partition(g)
    rb, ri = oracle.partition(V, P, ref)
    assert np.array_equal(u32(b), rb)
    assert np.array_equal(inter.cpu().numpy().astype(np.uint64), ri)


@pytest.mark.parametrize("E", [0, 1, 31, 32, 33, 1024, 32767, 32768, 32769, 200001])
@pytest.mark.parametrize("share", [0.0, 0.5, 0.96, 1.0])
@pytest.mark.parametrize("off", [0, 1])
def test_compact_words_and_tiles(sssp, E, share, off):
    """E distinct edges exactly; kept with the given share; the mask at an aligned and an odd address
    (any non-zero byte keeps)."""
    V = 700
    rng = np.random.default_rng(E + int(100 * share))
    key = rng.choice(V * (V - 1), E, replace=False)
    src, dst = (key // (V - 1)).astype(np.uint32), (key % (V - 1)).astype(np.uint32)
    dst += dst >= src  # no loops
    w = rng.integers(1, 1000, E).astype(np.uint32)
    ref = oracle.csr(V, src, dst, w)
    assert ref.E == E
    g = sssp.build_csr(V, src, dst, w)
    keep = (rng.random(E) < share).astype(np.uint8) * rng.integers(1, 256, E).astype(np.uint8)
    buf = torch.zeros(E + 33, dtype=torch.uint8, device="cuda")
    at = (-buf.data_ptr()) % 16 + off
    buf[at:at + E] = torch.from_numpy(keep).cuda()
    gp = sssp.compact(g, buf[at:at + E])
    rp = oracle.compact(ref, (keep != 0).astype(np.uint8))
    assert gp.E == rp.E
    assert np.array_equal(u32(gp.row_ptr), rp.row_ptr)
    assert np.array_equal(u32(gp.col)[:gp.E], rp.col[:gp.E]) and np.array_equal(u32(gp.w)[:gp.E], rp.w[:gp.E])
    assert np.array_equal(u32(gp.eid)[:gp.E], np.flatnonzero(keep).astype(np.uint32))


def check_build(sssp, V, src, dst, w, **kw):
    ref = oracle.csr(V, src, dst, w)
    g = sssp.build_csr(V, src, dst, w, **kw)
    assert g.E == ref.E
    assert np.array_equal(u32(g.row_ptr), ref.row_ptr)
    E = g.E
    assert np.array_equal(u32(g.col)[:E], ref.col[:E])
    assert np.array_equal(u32(g.w)[:E], ref.w[:E].view(np.uint32))
    assert np.array_equal(u32(g.eid)[:E], first_of_least(src, dst, w, V))
    return g, ref


def first_of_least(src, dst, w, V):
    """Input index of every canonical edge: the lowest index among the least weights of its pair."""
    idx = np.flatnonzero(src != dst)
    order = idx[np.lexsort((idx, w[idx], dst[idx], src[idx]))]
    key = src[order].astype(np.uint64) * V + dst[order]
    return order[np.concatenate([[True], key[1:] != key[:-1]])].astype(np.uint32) if order.size else order.astype(np.uint32)


@pytest.mark.parametrize("V,E", [(V, E) for V in (2, 3, 17, 512, 513, 70000) for E in (1, 2, 4095, 4096, 4097, 12289, 150001)]
                         + [((1 << 26) + 5, 12289)])
def test_build_tiles_and_key_widths(sssp, V, E):
    """One to six digits, tiles of 4,096 pairs and their remainders, many repeated pairs (small V)."""
    src, dst, w = edges(V % 1000 + E, V, E, hi=7)
    src[-1:], dst[-1:] = V - 1, 0
    check_build(sssp, V, src, dst, w)


@pytest.mark.parametrize("f32", [False, True])
def test_build_runs_across_tiles(sssp, f32):
    """A run of equal pairs inside a warp, across warps, across one and several tiles, with its least
    weight first, last and in the middle, and ties."""
    rng = np.random.default_rng(3)
    V = 40
    for reps in (31, 700, 5000, 30000):
        src = np.concatenate([np.full(reps, 3), rng.integers(0, V, 9000), np.full(reps, 20), [39, 39]]).astype(np.uint32)
        dst = np.concatenate([np.full(reps, 5), rng.integers(0, V, 9000), np.full(reps, 7), [0, 0]]).astype(np.uint32)
        for least in (0, reps // 2, reps - 1):
            w = rng.integers(2, 6, src.size).astype(np.float32 if f32 else np.uint32)
            w[least] = 1
            w[reps + 9000 + least] = 1
            perm = rng.permutation(src.size)
            check_build(sssp, V, src[perm], dst[perm], w[perm])
            check_build(sssp, V, src, dst, w)


@pytest.mark.parametrize("gap", [0, 1, 15, 16, 17, 31, 33, 70, 5000, 1000003])
def test_build_rows_without_edges(sssp, gap):
    """Runs of rows without an edge before the first edge, between edges that are neighbours in a warp's step,
    in two steps and in two tiles, and after the last."""
    tails = np.concatenate([[gap], gap + 1 + np.arange(40) * (gap + 1)])
    V = int(tails[-1]) + 1 + gap + 1
    for reps in (1, 3, 200):  # edges of a row
        src = np.repeat(tails, reps).astype(np.uint32)
        dst = ((src + 1 + np.tile(np.arange(reps), tails.size)) % V).astype(np.uint32)
        check_build(sssp, V, src, dst, np.full(src.size, 7, np.uint32))


def test_build_without_an_edge_left_and_bad_edges_reported(sssp):
    v = np.arange(9000, dtype=np.uint32)
    g = sssp.build_csr(9000, v, v, np.ones(9000, np.uint32))  # loops only
    assert g.E == 0 and not u32(g.row_ptr).any()
    src, dst, w = edges(1, 100, 9000)
    for a, k, x in ((src, 5000, 100), (dst, 8999, 0xFFFFFFFF), (w, 4096, 0)):
        b = a.copy()
        b[k] = x
        with pytest.raises(sssp.SsspError):
            sssp.build_csr(100, *(b if y is a else y for y in (src, dst, w)))


@pytest.mark.parametrize("V,E,P", [(33, 4000, 2), (5000, 1023, 7), (5000, 1024, 7), (60001, 1025, 148), (60001, 900000, 1)])
def test_layout_ranges(sssp, V, E, P):
    """Ranges of 1,024 edges over empty rows, long rows and the last rows."""
    rng = np.random.default_rng(V + E)
    src, dst, w = edges(V + E, V, E)
    src[: E // 3] = rng.integers(0, 3, E // 3)
    ref = oracle.csr(V, src, dst, w)
    h = sssp.layout(sssp.build_csr(V, src, dst, w, partitions=P))
    ids, slots, lay = oracle.layout(ref, P)
    assert np.array_equal(u32(h.ids), ids) and np.array_equal(u32(h.slots), slots)
    assert np.array_equal(u32(h.row_ptr), lay.row_ptr)
    assert np.array_equal(u32(h.col)[:h.E], lay.col[:h.E]) and np.array_equal(u32(h.w)[:h.E], lay.w[:h.E])


def distinct_edges(rng, V, E, hubs=0):
    """Exactly E distinct edges without loops, the first `hubs` rows full."""
    key = np.concatenate([np.arange(hubs * V), rng.permutation(V * V) if V * V < 10 * E else rng.integers(0, V * V, 2 * E + 100)])
    key = key[key // V != key % V]
    _, at = np.unique(key, return_index=True)
    key = key[np.sort(at)][:E]
    assert key.size == E
    return (key // V).astype(np.uint32), (key % V).astype(np.uint32)


@pytest.mark.parametrize("V,E,hubs,P", [(40, 1, 0, 1), (40, 31, 0, 8), (40, 33, 0, 1), (300, 255, 0, 1), (300, 257, 0, 8),
                                        (300, 1025, 3, 1), (600, 8191, 9, 8), (600, 8193, 9, 9), (600, 8193, 9, 1),
                                        (1500, 60000, 35, 8), (1500, 60000, 35, 1), (20000, 2553599, 3, 64)])
@pytest.mark.parametrize("mode", [0, 1])
def test_prune_blocks_and_shares(sssp, V, E, hubs, P, mode):
    """Edge counts around a block's rounds (one round of 256 edges, of 1,024 edges and, from 2.5 M edges on,
    several), with rows of every length up to V - 1: pairs of many shares, and many pairs in a share."""
    if mode == 1 and E > 100000:
        V, E, hubs = 5000, 120000, 5
    rng = np.random.default_rng(E + P)
    src, dst = distinct_edges(rng, V, E, hubs)
    w = rng.integers(1, 60, E).astype(np.uint32)
    ref = oracle.csr(V, src, dst, w)
    g = sssp.build_csr(V, src, dst, w, partitions=P)
    keep, wit = sssp.prune(g, mode)
    rk, rw = oracle.trishla(ref, P, mode)
    assert np.array_equal(keep.cpu().numpy(), rk)
    assert np.array_equal(u32(wit), rw)


@pytest.mark.parametrize("V,P,deg", [(2100, 1, 2048), (2100, 1, 2049), (70000, 12, 3000), (70000, 148, 60000), (70000, 1, 30000),
                                     (5000, 2, 2047), (1025, 1025, 900)])
@pytest.mark.parametrize("f32", [False, True])
def test_layout_segments(sssp, V, P, deg, f32):
    """Rows whose edges to one partition are as long as a block holds (2,048), longer (sorted by the
    builder), and in several tiles; with rows of one edge between them."""
    rng = np.random.default_rng(V + deg)
    src, dst, w = edges(V, V, 5 * V)
    hub = np.concatenate([np.stack([np.full(deg, h), rng.choice(V - 1, deg, replace=False)]) for h in (V - 1, V // 2, 3)], axis=1)
    src, dst = np.concatenate([src, hub[0]]).astype(np.uint32), np.concatenate([dst, hub[1]]).astype(np.uint32)
    w = rng.uniform(0.5, 2.0, src.size).astype(np.float32) if f32 else rng.integers(1, 99, src.size).astype(np.uint32)
    ref = oracle.csr(V, src, dst, w)
    h = sssp.layout(sssp.build_csr(V, src, dst, w, partitions=P))
    ids, slots, lay = oracle.layout(ref, P)
    assert np.array_equal(u32(h.ids), ids) and np.array_equal(u32(h.slots), slots)
    assert np.array_equal(u32(h.row_ptr), lay.row_ptr)
    assert np.array_equal(u32(h.col)[:h.E], lay.col[:h.E])
    assert np.array_equal(u32(h.w)[:h.E], lay.w[:h.E].view(np.uint32))
    e = u32(h.eid)[:h.E]  # the edges of the graph that they were
    assert np.array_equal(np.sort(e), np.arange(h.E))
    assert np.array_equal(slots[ref.col[:h.E]][e], lay.col[:h.E]) and np.array_equal(ref.w[:h.E].view(np.uint32)[e], u32(h.w)[:h.E])


@pytest.mark.parametrize("P,deg,hubs,rest", [(1, 2048, 2, 60000), (1, 2049, 2, 60000), (2, 1300, 6, 60000), (1, 256, 500, 9000),
                                             (1, 257, 500, 9000), (1, 280, 500, 9000), (1, 330, 500, 9000), (1, 1500, 40, 40),
                                             (3, 4000, 9, 20)])
def test_layout_share_of_long_segments(sssp, P, deg, hubs, rest):
    """Long segments that are few of the edges (their heads are counted), or more than an eighth of them (the
    builder sorts)."""
    V = 5003
    rng = np.random.default_rng(deg + hubs)
    src, dst, w = edges(deg, V, rest)
    at = rng.choice(V, hubs, replace=False)
    src = np.concatenate([src] + [np.full(deg, h) for h in at]).astype(np.uint32)
    dst = np.concatenate([dst] + [rng.choice(np.delete(np.arange(V), h), deg, replace=False) for h in at]).astype(np.uint32)
    w = rng.integers(1, 99, src.size).astype(np.uint32)
    ref = oracle.csr(V, src, dst, w)
    h = sssp.layout(sssp.build_csr(V, src, dst, w, partitions=P))
    ids, slots, lay = oracle.layout(ref, P)
    assert np.array_equal(u32(h.ids), ids) and np.array_equal(u32(h.slots), slots)
    assert np.array_equal(u32(h.row_ptr), lay.row_ptr)
    assert np.array_equal(u32(h.col)[:h.E], lay.col[:h.E]) and np.array_equal(u32(h.w)[:h.E], lay.w[:h.E])
    e = u32(h.eid)[:h.E]
    assert np.array_equal(np.sort(e), np.arange(h.E)) and np.array_equal(slots[ref.col[:h.E]][e], lay.col[:h.E])


@pytest.mark.parametrize("what", ["order", "twice", "loop", "head", "weight"])
def test_layout_of_rows_that_are_not_canonical(sssp, what):
    """Rows out of order, repeated heads and loops go through the builder, as an edge list would; bad heads
    and weights are reported."""
    V, P = 3000, 7
    src, dst, w = edges(5, V, 8 * V)
    g = sssp.build_csr(V, src, dst, w, partitions=P)
    rp, col, wt = u32(g.row_ptr), u32(g.col)[:g.E].copy(), u32(g.w)[:g.E].copy()
    r = int(np.argmax(np.diff(rp.astype(np.int64))))
    a = int(rp[r])
    if what == "order":
        col[a], col[a + 1] = col[a + 1], col[a]
    elif what == "twice":
        col[a + 1] = col[a]
    elif what == "loop":
        col[a] = r
    elif what == "head":
        col[a] = V
    else:
        wt[a] = 0
    dev = lambda x: torch.from_numpy(x.view(np.int32)).cuda()
    h = sssp.DeviceGraph(V, g.E, dev(rp.copy()), dev(col), dev(wt), g.wtype, P)
    if what in ("head", "weight"):
        with pytest.raises(sssp.SsspError):
            sssp.layout(h)
        return
    out = sssp.layout(h)
    tails = np.repeat(np.arange(V), np.diff(rp.astype(np.int64))).astype(np.uint32)
    # the edge list renumbered by the ids that the layout found, through the oracle
    slots = u32(out.slots)
    want = oracle.csr(V, slots[tails], slots[col], wt)
    E = int(want.row_ptr[-1])
    assert np.array_equal(u32(out.row_ptr), want.row_ptr)
    assert np.array_equal(u32(out.col)[:E], want.col[:E]) and np.array_equal(u32(out.w)[:E], want.w[:E])
