"""The radix passes where they can go wrong: one key, the edges of a tile of
1024 and of 4096 keys, the size from which a sort takes the larger tile, sorts
of one to five passes, digit counts made anew after repeats are dropped, a run
of equal times too long to order in place (the sort by all three keys), and an
inverse permutation past the size up to which the last pass writes it, where the
pair tables take their larger tiles too.  Every
array of the temporal CSR equals the oracle's definition; for the last, that
definition's properties (whole numbers, no tolerance)."""
import numpy as np
import pytest

from test_gpu_csr import check_csr

pytestmark = pytest.mark.gpu


def _edges(n, m, t_hi, seed=1):
    rng = np.random.default_rng(seed)
    s = rng.integers(0, n, m).astype(np.uint32)
    d = ((s + 1 + rng.integers(0, n - 1, m)) % n).astype(np.uint32)
    return s, d, rng.integers(0, t_hi, m).astype(np.int64)


@pytest.fixture(scope="module")
def tg():
    import paper_2507_20441_gb300 as tg
    tg.build()
    return tg


@pytest.mark.parametrize("m", [1, 2, 31, 1023, 1024, 1025, 4095, 4097, 299_999, 300_001, 610_305])
def test_sizes(tg, oracle_mod, m):
    s, d, _ = _edges(1000, m, 2)
    t = np.random.default_rng(m).permutation(m).astype(np.int64)     # distinct times: no repeats
    check_csr(tg, oracle_mod, 1000, s, d, t)


@pytest.mark.parametrize("n,t_hi", [(2, 3), (127, 1 << 7), (129, 1 << 14), (1 << 15, 1 << 22), (1 << 22, (1 << 32) - 1)])
def test_digits_and_repeats(tg, oracle_mod, n, t_hi):
    s, d, t = _edges(n, 40_000, t_hi, n)
    s, d, t = (np.concatenate([x, x[:500]]) for x in (s, d, t))
    t[0], t[1] = 0, t_hi - 1
    check_csr(tg, oracle_mod, n, s, d, t, dedup=True)


@pytest.mark.parametrize("m", [20_000, 400_000])
def test_long_run_of_equal_times(tg, oracle_mod, m):
    s, d, t = _edges(900, m, 3)
    check_csr(tg, oracle_mod, 900, s, d, t, dedup=True)


def test_inverse_of_a_large_sort(tg):
    n, m = 70_001, 16_000_001
    s, d, _ = _edges(n, m, 2)
    t = np.random.default_rng(2).permutation(m).astype(np.int64)
    ctx = tg.Context()
    ctx.load_graph(n, s, d, t)
    at = np.arange(m, dtype=np.uint32)
    g_src, g_dst, g_t = ctx.edges()
    assert np.array_equal(g_t, at)                                   # the times are 0 .. m - 1
    for gid, pos, owner, g_owner in (("out_gid", "out_pos", "out_src", g_src), ("in_gid", "in_pos", "in_dst", g_dst)):
        gid, pos, owner = ctx.csr(gid), ctx.csr(pos), ctx.csr(owner)
        assert np.array_equal(pos[gid], at)
        assert np.array_equal(owner, g_owner[gid])
        assert np.all((owner[1:] > owner[:-1]) | ((owner[1:] == owner[:-1]) & (gid[1:] > gid[:-1])))
    # the pair tables (larger tiles than a small array's)
    pairs, count = np.unique(g_src.astype(np.int64) * n + g_dst, return_counts=True)
    start = np.concatenate([[0], np.cumsum(count)])
    assert np.array_equal(ctx.csr("pair_dst"), pairs % n)
    assert np.array_equal(ctx.csr("pair_off"), start)
    assert np.array_equal(ctx.csr("vpair_off"), np.searchsorted(pairs // n, np.arange(n + 1)))
    own = np.zeros((m // 32 + 1) * 32, np.uint8)
    own[start[:-1]] = 1
    assert np.array_equal(ctx.csr("own_multi"), np.packbits(own, bitorder="little").view(np.uint32))
    ctx.close()
