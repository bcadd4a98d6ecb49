"""Window totals and their running sum at the edges of a tile (1024 windows, of
both layers together and of one) and past one step of the look-back (32 tiles):
W, every total and the samples, which read the sums and the guide tables' offsets,
equal the oracle's (whole numbers, no tolerance)."""
import numpy as np
import pytest

from helpers import oracle_result

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nwin", [1, 511, 512, 513, 1023, 1024, 1025, 33 * 512 + 1])
def test_totals_equal_the_oracle(oracle_mod, nwin):
    import paper_2507_20441_gb300 as tg
    tg.build()
    rng = np.random.default_rng(nwin)
    n, delta = 12, 8
    # bursts of 1 to 6 edges, each alone in its window of either layer
    sizes = rng.integers(1, 7, nwin)
    m = int(sizes.sum())
    t = np.repeat(np.arange(nwin, dtype=np.int64) * 4 * delta - np.cumsum(sizes) + sizes, sizes) + np.arange(m)
    src = rng.integers(0, n, m).astype(np.uint32)
    dst = ((src + 1 + rng.integers(0, n - 1, m)) % n).astype(np.uint32)
    edges, tree, root = [(0, 1), (1, 2)], [0, 1], 0
    ctx = tg.Context()
    ctx.load_graph(n, src, dst, t)
    mo = ctx.motif(3, edges, [0, 1], delta).set_tree(tree, root)
    G = oracle_mod.Graph(n, src, dst, t)
    want = oracle_result(G, 3, edges, [0, 1], delta, tree, root, 2000, 4)
    assert mo.weights() == want[0]
    assert np.array_equal(mo.window_totals(), G.window_totals())
    r = mo.sample(2000, 4)
    assert (r.W, r.hits2, r.valid, r.rej_vertex, r.rej_delta, r.rej_order) == want
    ctx.close()
