"""The tree backward at the sizes where its warps change shape: sources that do not divide a warp's 32
items, more of them than a warp, vertices around a tile of 32, one source many times (every lane on one
tree edge), and trees that are one long path, against the oracle's sums.

Bound: the gradient is a float64 sum rounded to float32 once.  It has at most S * V terms, whose partial
sums stay below A = sum |g|, so the error is at most S * V * 2^-53 * A, and 2^-24 of the result."""
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


def check(sssp, V, src, dst, w, sources):
    ref = oracle.csr(V, src, dst, w)
    g = sssp.upload_csr(ref.V, ref.row_ptr, ref.col, ref.w, partitions=3)
    pred = sssp.solve(g, np.asarray(sources, np.uint32))[1]
    S = len(sources)
    gup = gg.normal_f32(S + V, (S, V))
    grad = sssp.backward(g, pred, torch.from_numpy(gup).cuda()).cpu().numpy().astype(np.float64)
    trees = [oracle.dijkstra(ref, int(s)) for s in sources]
    want = oracle.tree_grad(ref, np.stack([t[0] for t in trees]), np.stack([t[1] for t in trees]), gup)
    bound = S * V * 2.0**-53 * np.abs(gup.astype(np.float64)).sum() + 2.0**-24 * np.abs(want)
    assert (np.abs(grad - want) <= bound).all()
    assert (grad[want == 0] == 0).all()


@pytest.mark.parametrize("S", [1, 2, 3, 7, 31, 32, 33, 65])
@pytest.mark.parametrize("V", [31, 33, 1000])
def test_sources_and_vertices(sssp, S, V):
    rng = np.random.default_rng(S * V)
    E = 6 * V
    src, dst = rng.integers(0, V, E).astype(np.uint32), rng.integers(0, V, E).astype(np.uint32)
    check(sssp, V, src, dst, rng.uniform(0.5, 2.0, E).astype(np.float32), rng.integers(0, V, S).tolist())


@pytest.mark.parametrize("S", [5, 32, 40])
def test_one_source_many_times(sssp, S):
    rng = np.random.default_rng(S)
    src, dst = rng.integers(0, 700, 5000).astype(np.uint32), rng.integers(0, 700, 5000).astype(np.uint32)
    check(sssp, 700, src, dst, rng.uniform(0.5, 2.0, 5000).astype(np.float32), [9] * S)


@pytest.mark.parametrize("S", [1, 33])
def test_paths(sssp, S):
    V = 1500
    src = np.arange(V - 1, dtype=np.uint32)
    check(sssp, V, src, src + 1, np.random.default_rng(2).uniform(0.5, 2.0, V - 1).astype(np.float32), list(range(S)))


@pytest.mark.parametrize("S", [1, 2, 8, 9, 16, 17, 33, 47])
@pytest.mark.parametrize("kind", ["grid", "star"])
def test_deep_trees_and_many_children(sssp, S, kind):
    """Walks of many steps, whose warps take other leaves meanwhile; and one parent of most vertices.  Blocks of
    sixteen sources and their remainders."""
    rng = np.random.default_rng(S)
    if kind == "grid":
        at = np.arange(60 * 55).reshape(60, 55)
        a = np.concatenate([at[1:].ravel(), at[:, 1:].ravel()])
        b = np.concatenate([at[:-1].ravel(), at[:, :-1].ravel()])
    else:
        a, b = np.zeros(4000, np.int64), np.arange(1, 4001)
    src, dst = np.concatenate([a, b]).astype(np.uint32), np.concatenate([b, a]).astype(np.uint32)
    V = int(src.max()) + 1
    check(sssp, V, src, dst, rng.uniform(0.5, 2.0, src.size).astype(np.float32), rng.integers(0, V, S).tolist())
