"""A serving round that ran out of its wait may still be running when its query
has been told: the weights that its kernel reads are freed when it has ended, and
the context's next call starts from a stream with nothing of it left."""
import pytest

pytestmark = pytest.mark.gpu


class Watch:
    """Allocator hooks that keep every block to the end and note, for each one
    freed by the admission context, whether the main stream was idle."""

    def __init__(self):
        import torch
        import paper_2507_20441_gb300 as tg
        self.main, self.of, self.keep, self.busy_frees, self.frees = None, {}, [], 0, 0

        def _alloc(nbytes, stream, user):
            s = torch.cuda.ExternalStream(stream)
            if self.main is None:
                self.main = s
            with torch.cuda.stream(s):
                t = torch.empty((nbytes,), dtype=torch.uint8, device="cuda")
            self.keep.append(t)
            self.of[t.data_ptr()] = stream
            return t.data_ptr()

        def _free(ptr, nbytes, stream, user):
            if self.of.pop(ptr) != self.main.cuda_stream:
                self.frees += 1
                self.busy_frees += not self.main.query()

        self.hooks = (tg.ALLOC_FN(_alloc), tg.FREE_FN(_free))


@pytest.mark.parametrize("how", ["stop", "evict"])
def test_weights_outlive_a_late_round(how):
    import paper_2507_20441_gb300 as tg
    from paper_2507_20441_gb300 import synth
    tg.build()
    gr = synth.chung_lu_bursty(20_000, 400_000, 2.1, 6_000_000, seed=21)
    w = Watch()
    ctx = tg.Context(alloc_hooks=w.hooks)
    ctx.load_graph(gr.n, gr.src, gr.dst, gr.t)
    c4, c3 = synth.cycle(4, 86_400), synth.cycle(3, 86_400)
    # one motif's weights at a time, rounds of up to 2.6e8 samples, 1 ms of wait for each
    ctx.serve_start(max_active=2, tile=65536, round_tiles=4000, poll_timeout_ms=1, weight_budget=1)
    t = ctx.submit(c4.nv, c4.edges, c4.rank, c4.delta, 260_000_000, 3)
    with pytest.raises(tg.TimestError) as e:
        ctx.poll(t, timeout_ms=120_000)
    assert e.value.code == tg.TM_E_TIMEOUT and not w.main.query()      # told, and still running
    if how == "evict":
        t = ctx.submit(c3.nv, c3.edges, c3.rank, c3.delta, 1000, 4)    # takes the room of the first
        try:
            ctx.poll(t, timeout_ms=120_000)
        except tg.TimestError as e:                                    # (its own round may take a millisecond)
            assert e.code == tg.TM_E_TIMEOUT
        assert ctx.serve_stats()["evictions"] == 1 and w.frees
    ctx.serve_stop()
    assert w.frees and w.busy_frees == 0
    ctx.load_graph(gr.n, gr.src, gr.dst, gr.t)
    mo = ctx.motif(c4.nv, c4.edges, c4.rank, c4.delta)
    assert mo.weights() > 0 and mo.sample(10_000, 1).valid > 0
    ctx.close()
