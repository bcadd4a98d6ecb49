"""Admission counts what a motif's weights will hold: with a budget one byte
below two motifs' blocks the first is evicted for the second; with exactly their
sum both stay, unless the windows are so short that they are counted before they
take room (admission then knows an upper bound)."""
import pytest

pytestmark = pytest.mark.gpu

QUERIES = [   # (nv, edges, order, delta)
    (4, [(0, 1), (1, 2), (2, 3), (3, 0)], [0, 1, 2, 3], 86_400),
    (3, [(0, 1), (1, 2), (2, 0)], [0, 1, 2], 60),            # 1e5 windows: counted first
    (6, [(i, i + 1) for i in range(5)], [0, 1, 2, 3, 4], 600),
]


@pytest.mark.parametrize("first,second", [(0, 1), (1, 2), (2, 0), (0, 2)])
def test_resident_weights_stay_inside_the_budget(first, second):
    import paper_2507_20441_gb300 as tg
    from paper_2507_20441_gb300 import synth
    tg.build()
    gr = synth.chung_lu_bursty(20_000, 400_000, 2.1, 6_000_000, seed=21)
    ctx = tg.Context()
    ctx.load_graph(gr.n, gr.src, gr.dst, gr.t)

    def serve(queries, budget):
        ctx.serve_start(max_active=2, weight_budget=budget)
        for q in queries:
            r = ctx.poll(ctx.submit(*q, 1000, 3), timeout_ms=120_000)
            assert r.W > 0
        st = ctx.serve_stats()
        ctx.serve_stop()
        return st["resident_bytes"], st["evictions"]

    a, b = (serve([QUERIES[i]], 1 << 40)[0] for i in (first, second))
    two = [QUERIES[first], QUERIES[second]]
    if 1 not in (first, second):
        assert serve(two, a + b) == (a + b, 0)
    assert serve(two, a + b - 1) == (b, 1)
    ctx.close()
