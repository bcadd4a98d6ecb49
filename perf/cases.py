"""The calls that this framework's speed is judged by.

Each case is one call, or the sequence of calls, that a program of a user
repeats: a whole estimate on new edges (load, temporal CSR, weights, samples),
the weight pass or the sampler alone on a resident graph, and the other public
calls on resident weights (batch, trace, group, listing, tree selection).

Graphs have the shape of ``synth.py``'s: a directed power law with bursts of
repeated pairs, or uniform; they are drawn on the GPU from the seed.  Every
result is a whole number, apart from the estimate W * hits2 / (2k), one
rounding of whole numbers that depend on the library's own random streams: so
there is no value in 64 bits to compare with other than these numbers, and
the module has no ``exact``.
"""
import math

import numpy as np
import torch

import paper_2507_20441_gb300 as tm
from paper_2507_20441_gb300 import synth

PATH4 = [(0, 1), (1, 2), (2, 3)]
# five motifs over the spanning path 0->1->2->3 (extra edges, pi positions)
GROUP = [([(3, 0)], [0, 1, 2, 3]), ([(0, 2)], [0, 2, 3, 1]), ([(1, 3)], [0, 1, 2, 3]),
         ([(3, 1)], [1, 2, 3, 0]), ([(3, 0), (0, 2)], [0, 2, 3, 4, 1])]


def listed():
    return [
        # a small data set: the whole estimate is launches and latency
        dict(name="estimate_20k_triangle", call="estimate", graph="uniform", n=1000, m=20_000, span=1_000_000,
             motif="triangle", nv=3, delta=10_000, k=100_000),
        # an ordinary one: the 2M-edge workload of bench.py
        dict(name="estimate_2m_cycle4", call="estimate", graph="power", n=100_000, m=2_000_000, span=30_000_000,
             motif="cycle", nv=4, delta=86_400, k=1_000_000),
        # raw tuples as they come from a log: repeats and self loops are dropped; odd sizes
        dict(name="estimate_raw_5m_star4", call="estimate", graph="power", n=200_003, m=5_000_011, span=40_000_003,
             motif="out_star", nv=4, delta=3_600, k=333_333, raw=True),
        # the largest: bench.py's default workload
        dict(name="estimate_50m_cycle5_chord", call="estimate", graph="power", n=2_000_000, m=50_000_000,
             span=100_000_000, motif="cycle5_chord", nv=5, delta=3_600, k=10_000_000),
        # a new motif on a resident graph: the weight pass alone, a deep tree
        dict(name="weights_10m_path6", call="weights", graph="power", n=400_000, m=10_000_000, span=20_000_000,
             motif="path", nv=6, delta=3_600),
        # an interactive query on resident weights: one small launch
        dict(name="sample_2m_10k", call="sample", graph="power", n=100_000, m=2_000_000, span=30_000_000,
             motif="cycle", nv=4, delta=86_400, k=10_000),
        # many samples over long candidate lists (hubs, one day)
        dict(name="sample_10m_star5_3m", call="sample", graph="power", n=400_000, m=10_000_000, span=20_000_000,
             motif="in_star", nv=5, delta=86_400, k=3_000_000),
        # many queries in one launch: the pool of bench.py and the serving loop
        dict(name="batch_2m_32", call="batch", graph="power", n=100_000, m=2_000_000, span=30_000_000, queries=32,
             k=10_000_000),
        # every sample's tree, outcome and contribution, copied to the host
        dict(name="trace_2m_500k", call="trace", graph="power", n=100_000, m=2_000_000, span=30_000_000,
             motif="cycle", nv=4, delta=86_400, k=500_000),
        # five related motifs from one stream of samples
        dict(name="group_2m_1m", call="group", graph="power", n=100_000, m=2_000_000, span=30_000_000, nv=4,
             delta=86_400, k=1_000_000),
        # the motif instances behind the samples, on a dense graph with many of them
        dict(name="list_20k_300k", call="list", graph="uniform", n=100, m=20_000, span=1_000_000, motif="triangle",
             nv=3, delta=100_000, k=300_000),
        # tree and root selection: a weight pass for each candidate
        dict(name="select_2m_cycle5_chord", call="select", graph="power", n=100_000, m=2_000_000, span=30_000_000,
             motif="cycle5_chord", nv=5, delta=3_600, n_c=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["estimate"] * 5 + ["weights"] * 3 + ["sample"] * 3 + ["batch", "trace", "group", "list", "select"])
    top = {"estimate": 30e6, "weights": 30e6, "sample": 30e6, "batch": 2e6, "trace": 5e6, "group": 10e6, "list": 2e6,
           "select": 2e6}[call]
    m = _log(rng, 20_000, top)
    n = max(100, int(m / rng.uniform(16, 30)))
    c = dict(call=call, graph=rng.choice(["power", "power", "uniform"]), n=n, m=m,
             span=max(100_000, int(m / rng.uniform(0.02, 0.5))))
    if call == "batch":
        c.update(queries=rng.randint(2, 32), k=_log(rng, 20_000, 5_000_000))
        return c
    c["motif"] = rng.choice(["triangle", "path", "cycle", "out_star", "in_star", "cycle5_chord"])
    c["nv"] = {"triangle": 3, "cycle5_chord": 5}.get(c["motif"]) or rng.randint(3, 5 if call == "select" else 6)
    c["delta"] = rng.choice([600, 3_600, 86_400, _log(rng, 300, 100_000)])
    # a day's window over a graph this dense would make one pass outlast the largest listed one
    if m > 1e7:
        c["delta"] = min(c["delta"], 10_000)
    if call == "estimate" and rng.random() < 0.3:
        c["raw"] = True
    if call == "group":
        c["nv"] = 4
        del c["motif"]
    if call in ("estimate", "sample"):
        c["k"] = _log(rng, 1_000, 4_000_000)
    elif call in ("trace", "list"):
        c["k"] = _log(rng, 1_000, 1_000_000)
    elif call == "group":
        c["k"] = _log(rng, 1_000, 2_000_000)
    elif call == "select":
        c["n_c"] = rng.randint(1, 3)
    return c


# ---- inputs ---------------------------------------------------------------
def _endpoints(gen, count, n, power):
    u = torch.rand(count, generator=gen, device="cuda", dtype=torch.float64)
    if power:   # weight (i + 1)^(-10/11) (gamma = 2.1): the inverse of its integral
        u = (u * ((n + 1.0) ** (1 / 11) - 1) + 1) ** 11 - 1
    else:
        u = u * n
    return u.long().clamp_(0, n - 1)


def _mix(x):
    x = x * -7046029254386353131
    x = x ^ (x >> 29)
    x = x * -4658895280553007687
    return x ^ (x >> 32)


def _edges(case, seed):
    """src, dst (int32 holding u32 ids) and t (int64) on the GPU: unique tuples in no order, or raw ones."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n, m, span, raw = case["n"], case["m"], case["span"], case.get("raw", False)
    power = case["graph"] == "power"
    want = m if raw else m + m // 20 + 100      # some more: repeats are dropped
    rep = int(want * 0.3) if power else 0       # re-emissions of an earlier pair, about ten minutes later
    base = want - rep
    u, v = _endpoints(gen, base, n, power), _endpoints(gen, base, n, power)
    v = torch.where(u == v, (v + 1) % n, v)
    t = torch.randint(0, span, (base,), generator=gen, device="cuda")
    if rep:
        pick = torch.randint(0, base, (rep,), generator=gen, device="cuda")
        gap = torch.rand(rep, generator=gen, device="cuda", dtype=torch.float64).clamp_(min=1e-12).log_().mul_(-600.0)
        u, v = torch.cat([u, u[pick]]), torch.cat([v, v[pick]])
        t = torch.cat([t, (t[pick] + gap.ceil_().long().clamp_(min=1)).clamp_(max=span - 1)])
    if raw:     # one tuple in a hundred twice, one in two hundred a self loop
        at = torch.randint(0, m, (m // 100,), generator=gen, device="cuda")
        k = at.numel() // 2
        v[at[:k]] = u[at[:k]]
        frm = torch.arange(k, device="cuda")
        u[m - k:], v[m - k:], t[m - k:] = u[frm].clone(), v[frm].clone(), t[frm].clone()
        order = torch.randperm(m, generator=gen, device="cuda")
    else:       # sorted by a hash of the tuple: repeats meet, and the order says nothing
        h, order = _mix((u * n + v) ^ _mix(t + 1)).sort()
        keep = torch.ones_like(h, dtype=torch.bool)
        keep[1:] = h[1:] != h[:-1]
        order = order[keep][:m]
    return u[order].int(), v[order].int(), t[order] + synth.T0


def _motif(case):
    nv, d = case["nv"], case["delta"]
    if case["motif"] == "triangle":
        return synth.triangle(d)
    if case["motif"] == "cycle5_chord":
        return synth.cycle5_chord(d)
    if case["motif"] == "path":
        return synth.path(nv, d)
    if case["motif"] == "cycle":
        return synth.cycle(nv, d)
    edges = [(0, i) if case["motif"] == "out_star" else (i, 0) for i in range(1, nv)]
    return synth.Motif(case["motif"], nv, edges, list(range(nv - 1)), d)


class State:
    def __init__(self, case, seed):
        self.case, self.seed = case, seed % (1 << 31)
        self.edges = _edges(case, self.seed)
        self.flags = tm.TM_DEVICE | (tm.TM_DEDUP | tm.TM_DROP_SELF if case.get("raw") else 0)
        self.ctx = ctx = tm.Context(device=0)
        call = case["call"]
        if call == "estimate":
            self.motifs = [self.handle(_motif(case))]
            return
        self.load()
        self.edges = None
        if call == "select":
            return
        if call == "batch":
            pool = synth.motif_pool(seed=7, count=case["queries"], k_lo=1e4, k_hi=case["k"])
            self.motifs = [self.handle(mo) for mo in pool]
            self.ks = [mo.k for mo in pool]
            self.seeds = [1000 * self.seed + i for i in range(len(pool))]
        elif call == "group":
            self.motifs = [ctx.motif(4, PATH4 + extra, order, case["delta"]).set_tree([0, 1, 2], 1)
                           for extra, order in GROUP]
        else:
            self.motifs = [self.handle(_motif(case))]
        if call == "weights":
            return
        for mo in self.motifs[:1] if call == "group" else self.motifs:
            mo.weights()

    def handle(self, mo):
        return self.ctx.motif(mo.nv, mo.edges, mo.rank, mo.delta)

    def load(self):
        self.ctx.load_graph(self.case["n"], *self.edges, flags=self.flags)

    def __del__(self):
        ctx = getattr(self, "ctx", None)
        if ctx is not None:
            ctx.close()


def prepare(case, seed):
    return State(case, seed)


# ---- one pass -------------------------------------------------------------
def _numbers(r):
    return {"W": r.W, "hits2": r.hits2, "counts": np.array([r.k, r.valid, r.rej_vertex, r.rej_delta, r.rej_order]),
            "estimate": r.estimate}


def _table(rs):
    return {"numbers": np.array([[r.W, r.hits2, r.k, r.valid, r.rej_vertex, r.rej_delta, r.rej_order] for r in rs]),
            "estimate": np.array([r.estimate for r in rs])}


def run(state):
    case, ctx = state.case, state.ctx
    call, seed = case["call"], state.seed
    if call == "estimate":
        state.load()
        mo = state.motifs[0]
        mo.weights()
        return {"m": ctx.m, "t_min": ctx.t_min, "T": ctx.T, **_numbers(mo.sample(case["k"], seed))}
    if call == "weights":
        mo = state.motifs[0]
        return {"W": mo.weights(), "windows": mo.window_totals().view(np.int64)}
    if call == "sample":
        return _numbers(state.motifs[0].sample(case["k"], seed))
    if call == "batch":
        return _table(ctx.batch_run(state.motifs, state.ks, state.seeds))
    if call == "trace":
        r, gids, contrib, reason = state.motifs[0].sample_trace(case["k"], seed)
        return {"gids": gids.view(np.int32), "contrib": contrib.view(np.int64), "reason": reason, **_numbers(r)}
    if call == "group":
        return _table(ctx.sample_group(state.motifs, case["k"], seed))
    if call == "list":
        gids, ids, total = state.motifs[0].sample_list(case["k"], seed, max_inst=200_000)
        # the call's buffers of max_inst rows, of which the first min(total, max_inst) are filled
        return {"gids": gids.base.view(np.int32), "ids": ids.base.view(np.int64), "total": total}
    mo = _motif(case)
    best, cands = ctx.select_tree(mo.nv, mo.edges, mo.rank, mo.delta, n_c=case["n_c"])
    order, parent = best.plan()
    best.free()
    return {"order": order, "parent": parent, "W": np.array([c["W"] for c in cands]),
            "root": np.array([c["root"] for c in cands]), "tree": np.array([c["tree_mask"] for c in cands])}


def work(case):
    """Bytes alone: the arithmetic is whole numbers.  16 for each edge tuple read; on a resident graph 12 for each
    edge (time and endpoints); for each sample 12 for each edge of its tree, and the records that a call returns."""
    m, nv, k, call = case["m"], case.get("nv", 5), case.get("k", 0), case["call"]
    if call == "estimate":
        return {"bytes": 16 * m + 12 * (nv - 1) * k, "flops": 0}
    if call == "weights":
        return {"bytes": 12 * m + 8 * (case["span"] // case["delta"] + 1), "flops": 0}
    if call == "select":
        return {"bytes": 12 * m * (nv - 1) * case["n_c"], "flops": 0}
    if call == "batch":
        pool = synth.motif_pool(seed=7, count=case["queries"], k_lo=1e4, k_hi=case["k"])
        return {"bytes": sum(12 * (mo.nv - 1) * mo.k for mo in pool), "flops": 0}
    out = {"trace": 4 * (nv - 1) + 12}.get(call, 0)
    return {"bytes": (12 * (nv - 1) + out) * k, "flops": 0}
