"""tm_select_tree has nothing left to run when it returns: the stream is idle and
the winner's guide tables are counted in the root phase."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_c,all_roots", [(1, False), (2, True)])
def test_selection_ends_before_it_returns(n_c, all_roots):
    import torch
    import paper_2507_20441_gb300 as tg
    from paper_2507_20441_gb300 import synth
    tg.build()
    gr = synth.chung_lu_bursty(100_000, 2_000_000, 2.1, 30_000_000, seed=2)
    stream = torch.cuda.Stream()
    ctx = tg.Context(stream=stream.cuda_stream, profile=1)
    ctx.load_graph(gr.n, gr.src, gr.dst, gr.t)
    mo = synth.cycle5_chord(3600)
    for _ in range(3):
        ctx.phase_times()
        best, cands = ctx.select_tree(mo.nv, mo.edges, mo.rank, mo.delta, n_c=n_c, all_roots=all_roots)
        assert stream.query()
        ms, launches = ctx.phase_times()["root"]
        assert launches == 2 * len(cands) + 1 and ms > 0      # scan and totals each, one fill
        best.free()
    ctx.close()
