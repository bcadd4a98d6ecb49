"""The window pass (Constraint 3, Alg. 1) at the edges of its tiles and at window
units from one time step to the whole span: units so short that the windows are
counted before they take room, and longer ones whose arrays are sized by what
the span allows.  W, every window total and the samples equal the oracle's
(whole numbers, no tolerance)."""
import numpy as np
import pytest

from helpers import oracle_result

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 31, 33, 2047, 2048, 2049, 40_000])
@pytest.mark.parametrize("delta", [1, 2, 700, 10_000_000])
def test_windows_equal_the_oracle(oracle_mod, m, delta):
    import paper_2507_20441_gb300 as tg
    tg.build()
    rng = np.random.default_rng(m + delta)
    n = 40
    src = rng.integers(0, n, m).astype(np.uint32)
    dst = ((src + 1 + rng.integers(0, n - 1, m)) % n).astype(np.uint32)
    t = np.cumsum(rng.integers(0, 5, m)).astype(np.int64) + np.arange(m)   # gaps of 1 to 5: some windows empty
    edges, tree, root = [(0, 1), (1, 2)], [0, 1], 0
    ctx = tg.Context()
    ctx.load_graph(n, src, dst, t)
    mo = ctx.motif(3, edges, [0, 1], delta).set_tree(tree, root)
    G = oracle_mod.Graph(n, src, dst, t)
    if delta > m:      # the oracle lists the candidates of every edge: whole lists here
        G.set_motif(2, [(0, 1)], [0], delta, [0], 0)
        mo = ctx.motif(2, [(0, 1)], [0], delta)
        assert mo.weights() == G.weights()
        assert np.array_equal(mo.window_totals(), G.window_totals())
        return
    want = oracle_result(G, 3, edges, [0, 1], delta, tree, root, 3000, 4)
    assert mo.weights() == want[0]
    assert np.array_equal(mo.window_totals(), G.window_totals())
    r = mo.sample(3000, 4)
    assert (r.W, r.hits2, r.valid, r.rej_vertex, r.rej_delta, r.rej_order) == want
    ctx.close()
