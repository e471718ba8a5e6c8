"""The one-time graph steps at the sizes where their kernels change path: partition counts up to a
vertex each (ranges that cross many partitions, empty ones among them), compaction around its mask
words and tiles and with an unaligned keep mask, all against the CPU oracle (integers: equal)."""
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
