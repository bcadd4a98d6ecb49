"""Weight passes that exceed 2^64 and what comes after them: TM_E_OVERFLOW, no
write outside the blocks that the allocator gave (each is followed by a strip
that has to keep its pattern), the same results as before from motifs that were
there, and a tree selection whose last candidate overflowed."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PAD = 4 << 20


class Strips:
    """Allocator hooks: every block is followed by PAD bytes of a pattern."""

    def __init__(self):
        import torch
        import paper_2507_20441_gb300 as tg
        self.live, self.broken = {}, 0

        def _alloc(nbytes, stream, user):
            t = torch.empty(nbytes + PAD, dtype=torch.uint8, device="cuda")
            t[nbytes:] = 0xA5
            torch.cuda.synchronize()
            self.live[t.data_ptr()] = (t, nbytes)
            return t.data_ptr()

        def _free(ptr, nbytes, stream, user):
            self.check()
            del self.live[ptr]

        self.hooks = (tg.ALLOC_FN(_alloc), tg.FREE_FN(_free))

    def check(self):
        import torch
        torch.cuda.synchronize()
        for t, nbytes in self.live.values():
            self.broken += int((t[nbytes:] != 0xA5).any())


def _star(hub):
    """The out-edges of a hub, at distinct times."""
    return np.zeros(hub, np.uint32), np.arange(1, hub + 1, dtype=np.uint32), np.arange(hub, dtype=np.int64)


# 740: just below 2^64; from 2375 on the wrapped totals are far below the sums before them
@pytest.mark.parametrize("hub", [740, 2000, 2375, 3000, 8192])
def test_overflow_stays_inside_its_blocks(hub):
    import paper_2507_20441_gb300 as tg
    tg.build()
    pads = Strips()
    ctx = tg.Context(alloc_hooks=pads.hooks)
    ctx.load_graph(hub + 1, *_star(hub))
    pair = ctx.motif(3, [(0, 1), (0, 2)], [0, 1], 10_000)
    W = pair.weights()
    assert W == hub * (hub - 1) // 2
    want = pair.sample(5000, 3)
    star = ctx.motif(8, [(0, i) for i in range(1, 8)], list(range(7)), 10_000).set_tree(list(range(7)), 0)
    total = sum(i ** 6 for i in range(hub))       # the root edge and six later ones each
    for _ in range(2):
        if total >= 1 << 64:
            with pytest.raises(tg.TimestError) as e:
                star.weights()
            assert e.value.code == tg.TM_E_OVERFLOW
        else:
            assert star.weights() == total
        pads.check()
        got = pair.sample(5000, 3)
        assert (got.W, got.hits2, got.valid, got.rej_vertex, got.rej_delta, got.rej_order) == \
               (want.W, want.hits2, want.valid, want.rej_vertex, want.rej_delta, want.rej_order)
    again = ctx.motif(3, [(0, 1), (0, 2)], [0, 1], 10_000)
    assert again.weights() == W
    assert again.sample(5000, 3).hits2 == want.hits2
    assert pads.broken == 0
    ctx.close()


@pytest.mark.parametrize("behind", [0, 1, 3])
@pytest.mark.parametrize("later", [8192, 8191])
def test_a_partial_product_that_wraps_to_zero(later, behind):
    """The root edge h->v has five children at h (8192 candidates each: 2^65, which
    is 0 in 64 bits) and one at v: an overflow, unless nothing follows at v."""
    import paper_2507_20441_gb300 as tg
    tg.build()
    h, v = 0, 1
    src = np.concatenate([[h], np.zeros(later), np.full(behind, v)]).astype(np.uint32)
    dst = np.concatenate([[v], np.arange(later) + 2, np.arange(behind) + 2]).astype(np.uint32)
    t = np.arange(src.size, dtype=np.int64)
    ctx = tg.Context()
    ctx.load_graph(later + 2, src, dst, t)
    edges = [(0, 1)] + [(0, i) for i in range(2, 7)] + [(1, 7)]
    mo = ctx.motif(8, edges, list(range(7)), 100_000).set_tree(list(range(7)), 0)
    if later ** 5 * behind >= 1 << 64:
        with pytest.raises(tg.TimestError) as e:
            mo.weights()
        assert e.value.code == tg.TM_E_OVERFLOW
    else:
        assert mo.weights() == later ** 5 * behind
    ctx.close()


def test_selection_ending_in_an_overflow():
    """A hub with 25,000 out-edges and chains between its first neighbours: the
    star over the hub overflows, trees that use a chain do not.  A selection whose
    last candidate overflows returns the winner with its guide tables filled: it
    samples like a motif pinned to its tree."""
    import paper_2507_20441_gb300 as tg
    tg.build()
    hub = 25_000
    a = np.repeat(np.arange(1, 41), 10)           # ten edges each 1->2, 2->3, ..., later and later
    src = np.concatenate([np.zeros(hub, np.int64), a]).astype(np.uint32)
    dst = np.concatenate([np.arange(1, hub + 1), a + 1]).astype(np.uint32)
    t = np.arange(hub + a.size, dtype=np.int64)
    ctx = tg.Context()
    ctx.load_graph(hub + 1, src, dst, t)
    nv, edges = 6, [(0, i) for i in range(1, 6)] + [(i, i + 1) for i in range(1, 5)]
    args = (nv, edges, list(range(9)), 100_000)
    ranked = len(tg.tm_tree_candidates(*args[:3]))
    best, cands = ctx.select_tree(*args, n_c=ranked, all_roots=False)
    status = [c["status"] for c in cands]
    assert tg.TM_E_OVERFLOW in status and tg.TM_OK in status
    best.free()
    tried = 0
    for n_c in range(2, ranked + 1):
        ok = [i for i in range(n_c) if status[i] == tg.TM_OK]
        if status[n_c - 1] != tg.TM_E_OVERFLOW or not ok:
            continue
        win = min(ok, key=lambda i: (cands[i]["W"], i))
        if cands[win]["W"] == 0:
            continue
        tree = [e for e in range(32) if cands[win]["tree_mask"] >> e & 1]
        best, _ = ctx.select_tree(*args, n_c=n_c, all_roots=False)
        pinned = ctx.motif(*args).set_tree(tree, cands[win]["root"])
        assert pinned.weights() == cands[win]["W"]
        x, y = best.sample(20_000, 7), pinned.sample(20_000, 7)
        assert (x.W, x.hits2, x.valid, x.rej_vertex, x.rej_delta, x.rej_order) == \
               (y.W, y.hits2, y.valid, y.rej_vertex, y.rej_delta, y.rej_order)
        best.free(); pinned.free()
        tried += 1
        if tried == 5:
            break
    assert tried
    ctx.close()
