"""Candidate ranges that the weight pass does not keep (16,383 entries and more):
one entry below and above, long in one layer and short in the other, met by leaf
children, by children with children and by both; and ranges whose numbers of
candidates are not known either (a weight block without ranges is tested with
the allocator's refusals).  A few edges into a hub with one long list, so that
the oracle, which lists every candidate, stays quick.  W, hits2, every counter
and every sampled tree equal the oracle's (whole numbers, no tolerance)."""
import numpy as np
import pytest

from helpers import oracle_result

pytestmark = pytest.mark.gpu

HUB = 0
# edges as seen along time for "later"; reversed in time and direction for "earlier"
MOTIFS = {
    "leaf": (3, [(0, 1), (1, 2)]),
    "inner": (4, [(0, 1), (1, 2), (2, 3)]),
    "both": (5, [(0, 1), (1, 2), (2, 3), (1, 4)]),
}


def _graph(times, roots, seed):
    """roots edges x -> hub, an edge hub -> y at each of `times`, one y -> z after each second of these."""
    rng = np.random.default_rng(seed)
    ny = 50
    y = rng.integers(1, ny, times.size)
    x = rng.integers(1, ny + 10, roots.size)                 # some x are a y too: excluded entries
    src = np.concatenate([x, np.full(times.size, HUB), y[::2]])
    dst = np.concatenate([np.full(roots.size, HUB), y, np.full(y[::2].size, ny + 20)])
    t = np.concatenate([roots, times, times[::2] + 1])
    return ny + 21, src, dst, t


def _check(tg, oracle_mod, n, src, dst, t, name, order, delta, c2):
    nv, edges = MOTIFS[name]
    ne = len(edges)
    rank = list(range(ne))
    if order == "earlier":       # time and every edge turned round
        src, dst, t = dst, src, t.max() - t
        edges = [(b, a) for a, b in edges]
        rank = rank[::-1]
    src, dst, t = src.astype(np.uint32), dst.astype(np.uint32), t.astype(np.int64)
    ctx = tg.Context()
    ctx.load_graph(n, src, dst, t, flags=tg.TM_DEDUP)
    G = oracle_mod.Graph(n, src, dst, t, flags=oracle_mod.DEDUP)
    want = oracle_result(G, nv, edges, rank, delta, range(ne), 0, 2000, 5, c2=c2)
    mo = ctx.motif(nv, edges, rank, delta).set_tree(list(range(ne)), 0).set_constraints(c2, True)
    assert want[0] > 0 and mo.weights() == want[0]
    r = mo.sample(2000, 5)
    assert (r.W, r.hits2, r.valid, r.rej_vertex, r.rej_delta, r.rej_order) == want
    _, gids, contrib, why = mo.sample_trace(500, 5)
    ro = G.sample(500, 5, trace=True)
    assert np.array_equal(gids, ro[1]) and np.array_equal(contrib, ro[2]) and np.array_equal(why, ro[3])
    ctx.close()


@pytest.fixture(scope="module")
def tg():
    import paper_2507_20441_gb300 as tg
    tg.build()
    return tg


@pytest.mark.parametrize("c2", [True, False])
@pytest.mark.parametrize("order", ["later", "earlier"])
@pytest.mark.parametrize("name", sorted(MOTIFS))
@pytest.mark.parametrize("entries", [16_382, 16_383, 16_384, 40_000])
def test_around_the_longest_kept_range(tg, oracle_mod, entries, name, order, c2):
    g = _graph(100 + 2 * np.arange(entries), np.arange(40), entries)
    _check(tg, oracle_mod, *g, name, order, 1_000_000, c2)


@pytest.mark.parametrize("order", ["later", "earlier"])
@pytest.mark.parametrize("name", sorted(MOTIFS))
def test_long_in_one_layer_or_both(tg, oracle_mod, name, order):
    # windows of two deltas, one starting every delta: ranges clipped in one layer, long or short there
    roots = np.random.default_rng(7).integers(40_500, 79_990, 40)
    g = _graph(40_000 + 2 * np.arange(40_000), roots, 3)
    _check(tg, oracle_mod, *g, name, order, 40_000, True)
