"""The windows and candidate ranges that the candidates of one tree selection
share: with windows counted before they take room (short deltas) and sized by the
span, the chosen motif samples like one pinned to its tree, before and after its
weights are taken again on their own."""
import pytest

from helpers import SMALL_MOTIFS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["cycle4", "bowtie", "cycle5_chord"])
@pytest.mark.parametrize("delta", [3, 600, 10_000_000_000])
def test_chosen_motif_equals_a_pinned_one(name, delta):
    import paper_2507_20441_gb300 as tg
    from paper_2507_20441_gb300 import synth
    tg.build()
    nv, edges, order = SMALL_MOTIFS[name]
    gr = synth.chung_lu_bursty(900, 20_001, 2.1, 400_000, seed=5)
    ctx = tg.Context()
    ctx.load_graph(gr.n, gr.src, gr.dst, gr.t)
    best, cands = ctx.select_tree(nv, edges, order, delta, n_c=3, all_roots=True)
    for c in cands:
        tree = [e for e in range(32) if c["tree_mask"] >> e & 1]
        mo = ctx.motif(nv, edges, order, delta).set_tree(tree, c["root"])
        if c["status"] == tg.TM_OK:
            assert c["W"] == mo.weights()
    win = min((i for i in range(len(cands)) if cands[i]["status"] == tg.TM_OK), key=lambda i: (cands[i]["W"], i))
    tree = [e for e in range(32) if cands[win]["tree_mask"] >> e & 1]
    pinned = ctx.motif(nv, edges, order, delta).set_tree(tree, cands[win]["root"])
    W = pinned.weights()
    for again in (False, True):
        if again:
            assert best.weights() == W
        if W:
            a, b = best.sample(5000, 7), pinned.sample(5000, 7)
            assert (a.W, a.hits2, a.valid, a.rej_vertex, a.rej_delta, a.rej_order) == \
                   (b.W, b.hits2, b.valid, b.rej_vertex, b.rej_delta, b.rej_order)
    ctx.close()
