"""Weights without kept candidate ranges: an allocator that has no room for a
motif's block with them, but for the block without, gives the same W, weights,
samples, traces, listings, groups, batches, served queries and selections, which
equal the oracle's (whole numbers, no tolerance)."""
import numpy as np
import pytest

from helpers import SMALL_MOTIFS, oracle_result, result_tuple

pytestmark = pytest.mark.gpu


class Sizes:
    """Allocator hooks over PyTorch's caching allocator that note the sizes
    asked for and refuse those in `refuse`."""

    def __init__(self):
        import torch
        import paper_2507_20441_gb300 as tg
        self.seen, self.refuse, self.refused = [], set(), 0

        def _alloc(nbytes, stream, user):
            self.seen.append(nbytes)
            if nbytes in self.refuse:
                self.refused += 1
                return None
            return int(torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0)))

        def _free(ptr, nbytes, stream, user):
            torch.cuda.caching_allocator_delete(int(ptr))

        self.hooks = (tg.ALLOC_FN(_alloc), tg.FREE_FN(_free))


PLANS = [   # (motif, tree, root, delta, Constraint 2, Constraint 3)
    ("cycle4", [0, 1, 2], 1, 86_400, True, True),
    ("cycle4", [0, 1, 2], 0, 86_400, True, True),
    ("cycle5_chord", [0, 1, 3, 4], 3, 20_000, True, True),
    ("out_star3", [0, 1, 2], 1, 86_400, True, True),
    ("path4_mixed", [0, 1, 2], 0, 600_000, False, True),
    ("bowtie", [0, 1, 3, 4], 0, 20_000, True, False),
]
K = 30_000


def _graph():
    from paper_2507_20441_gb300 import synth
    return synth.chung_lu_bursty(8000, 200_000, 2.1, 3_000_000, seed=8)


def _motif(ctx, plan):
    name, tree, root, delta, c2, c3 = plan
    return ctx.motif(*SMALL_MOTIFS[name], delta).set_tree(tree, root).set_constraints(c2, c3)


def _context(tg, gr):
    hook = Sizes()
    ctx = tg.Context(alloc_hooks=hook.hooks)
    ctx.load_graph(gr.n, gr.src, gr.dst, gr.t)
    for plan in PLANS:             # scratch grows to what they need
        _motif(ctx, plan).weights()
    return hook, ctx


def test_every_call_without_kept_ranges(oracle_mod):
    import paper_2507_20441_gb300 as tg
    tg.build()
    gr = _graph()
    all_hook, with_ranges = _context(tg, gr)
    hook, without = _context(tg, gr)
    G = oracle_mod.Graph(gr.n, gr.src, gr.dst, gr.t)
    for plan in PLANS:
        name, tree, root, delta, c2, c3 = plan
        nv, edges, rank = SMALL_MOTIFS[name]
        a, b = _motif(with_ranges, plan), _motif(without, plan)
        all_hook.seen.clear()
        W = a.weights()
        hook.refuse, hook.refused = set(all_hook.seen), 0
        assert b.weights() == W
        assert hook.refused == 1
        hook.refuse = set()
        want = oracle_result(G, nv, edges, rank, delta, tree, root, K, 5, c2=c2, c3=c3)
        assert want[0] == W and result_tuple(b.sample(K, 5)) == want
        for e in tree:
            for layer in (0, 1):
                assert np.array_equal(a.export_weights(e, layer), b.export_weights(e, layer))
        ta, tb = a.sample_trace(3000, 6), b.sample_trace(3000, 6)
        assert all(np.array_equal(x, y) for x, y in zip(ta[1:], tb[1:]))
        na = tg.tm_sample_noalloc(without.h, b.h, K, 5)
        assert result_tuple(na) == want
        la, lb = a.sample_list(5000, 7, max_inst=20_000), b.sample_list(5000, 7, max_inst=20_000)
        assert la[2] == lb[2] and np.array_equal(la[0], lb[0]) and np.array_equal(la[1], lb[1])
        ga, gb = (ctx.batch_run([m, m], [K, 777], [5, 8]) for ctx, m in ((with_ranges, a), (without, b)))
        assert [result_tuple(x) for x in ga] == [result_tuple(x) for x in gb]
        pa, pb = (ctx.sample_group([m, m], K, 5) for ctx, m in ((with_ranges, a), (without, b)))
        assert [result_tuple(x) for x in pa] == [result_tuple(x) for x in pb] == [want, want]
        a.free(); b.free()
    with_ranges.close(); without.close()


def test_selection_and_serving_without_kept_ranges():
    import paper_2507_20441_gb300 as tg
    gr = _graph()
    args = (*SMALL_MOTIFS["cycle5_chord"], 20_000)
    all_hook, with_ranges = _context(tg, gr)
    hook, without = _context(tg, gr)
    all_hook.seen.clear()
    best, cands = with_ranges.select_tree(*args, n_c=3)
    refuse = {max(all_hook.seen)}                  # the block that the candidates share
    all_hook.seen.clear()
    for c in cands:                                # and each candidate's own with ranges
        m = with_ranges.motif(*args).set_tree([e for e in range(6) if c["tree_mask"] >> e & 1], c["root"])
        m.weights()
        m.free()
    hook.refuse = refuse | set(all_hook.seen)
    got, cands2 = without.select_tree(*args, n_c=3)
    assert hook.refused >= len(cands) and cands2 == cands
    assert result_tuple(got.sample(K, 3)) == result_tuple(best.sample(K, 3))
    alone = with_ranges.motif(*args)
    all_hook.seen.clear()
    alone.weights()
    hook.refuse, hook.refused = set(all_hook.seen), 0
    without.serve_start(max_active=2)
    r = without.poll(without.submit(*args, K, 4), timeout_ms=120_000)
    st = without.serve_stats()
    without.serve_stop()
    assert hook.refused == 1 and st["completed"] == 1 and st["nomem_retries"] == 0
    assert result_tuple(r) == result_tuple(alone.sample(K, 4))
    with_ranges.close(); without.close()
