"""The persistent solve in the default policy on graphs that sssp_solve would sweep: warm starts with few tails, prunes
on idle time and the autotuner run it there.  Its kernel variants, hub widths and schedules against the CPU
oracle, bit for bit; that it ran is seen by the messages between its units, which a sweep has none of."""
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


def check(sssp, g, ref, sources, opts):
    opts.flags |= sssp.FLAG_TEST_PERSISTENT
    dist, pred, st, stats = sssp.solve(g, np.asarray(sources, np.uint32), opts, check=False)
    assert st == 0 and stats["remote_activations"] > 0
    for i, s in enumerate(sources):
        d, p, _ = oracle.dijkstra(ref, int(s))
        assert np.array_equal(u32(dist[i]), d.view(np.uint32)), f"dist, source {s}"
        assert np.array_equal(u32(pred[i]), p), f"pred, source {s}"


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("hubs", [0, 1, 48, 100000])
def test_hub_widths(sssp, f32, hubs):
    g0 = gg.rmat(gg.BASE_SEED + 640, 13, 16 << 13, wf32=(0.5, 2.0, 1e-4) if f32 else None)
    ref = oracle.csr_of(g0)
    h = sssp.layout(sssp.build_csr(g0.V, g0.src, g0.dst, g0.w, partitions=24))
    srcs = gg.pick_sources(gg.BASE_SEED + 640, g0, 3).tolist()
    for split in (1, 2):
        check(sssp, h, ref, srcs, sssp.options(delta=0.5 if f32 else 24, hub_count=hubs, split=split))


@pytest.mark.parametrize("seed", range(24))
def test_schedules(sssp, seed):
    rng = np.random.default_rng(4000 + seed)
    V, f32, lay = int(rng.integers(2000, 30000)), bool(seed % 2), bool(seed % 3 == 0)
    E = int(V * rng.integers(6, 14))
    src, dst = rng.integers(0, V, E).astype(np.uint32), rng.integers(0, V, E).astype(np.uint32)
    w = rng.uniform(0.5, 2.0, E).astype(np.float32) if f32 else rng.integers(1, 256, E).astype(np.uint32)
    ref = oracle.csr(V, src, dst, w)
    g = sssp.build_csr(V, src, dst, w, partitions=int(rng.integers(2, 149)))
    o = sssp.options(threads=int(rng.choice([128, 256, 512])), tile=int(rng.choice([32, 512, 1024, 4096])),
                     split=int(rng.integers(1, 4)), delta=float(rng.choice([0.05, 0.6, 3.0]) if f32 else rng.choice([4, 60, 300])),
                     blocks_per_sm=int(rng.integers(0, 3)), hub_count=int(rng.choice([0, 64])))
    check(sssp, sssp.layout(g) if lay else g, ref, rng.integers(0, V, int(rng.integers(1, 10))).tolist(), o)


def test_update_runs_it_too(sssp):
    rng = np.random.default_rng(9)
    V = 40000
    src, dst = rng.integers(0, V, 8 * V).astype(np.uint32), rng.integers(0, V, 8 * V).astype(np.uint32)
    w = rng.integers(2, 256, src.size).astype(np.uint32)
    at = rng.permutation(src.size)[:10000]
    w2 = w.copy()
    w2[at] //= 2
    sources = np.array([1, 2], np.uint32)
    dist, pred = sssp.solve(sssp.build_csr(V, src, dst, w, partitions=30), sources)[:2]
    dist, pred, st, stats = sssp.update(sssp.build_csr(V, src, dst, w2, partitions=30), dist, pred, src[at],
                                        sssp.options(flags=sssp.FLAG_TEST_PERSISTENT))
    assert st == 0 and stats["remote_activations"] > 0
    ref = oracle.csr(V, src, dst, w2)
    for i, s in enumerate(sources):
        d, p, _ = oracle.dijkstra(ref, int(s))
        assert np.array_equal(u32(dist[i]), d) and np.array_equal(u32(pred[i]), p)
