"""Performance cases of the px operators and pipelines on one GPU.

Each case is a piece of work a user of the library has it do, called through the
public entry points (the operator calls, the pipelines, the fused fragment
batches), with its input distributions and sizes taken from the workloads that the
tests and the benchmark define: scan-filter-aggregate over a columnar batch,
fact/dimension joins, the exchange-fed join and aggregation, late materialization
and batched fragments. `listed()` names fixed cases from the smallest calls to the
largest, `draw(rng)` gives one more of the same ranges, `prepare` makes a case's
inputs (on the GPU, from the seed alone) and the pipeline or buffers a program
keeps, `run` makes one pass and returns everything it computed, `work` gives the
bytes that pass cannot do without.

Every output is a whole number (int8, int32 or int64; sums wrap mod 2^64), so two
correct results are equal bit for bit and `exact` has nothing to add. Result
buffers are zeroed (or filled with the largest key) once when they are made: rows
past a result's device count are never written and compare equal.
"""
import math

import numpy as np
import torch

import paper_2606_24647_gb300 as px
from paper_2606_24647_gb300.pipelines import AtScalePipeline, JoinPipeline, PlainPipeline, WideJoinPipeline

DAYS = 2557                      # date domain: 7 years of day offsets
DATE_LO, DATE_HI = 895, 1662     # the join queries' date window, 30 % of the rows
SCAN_HI = 2506                   # the scan query keeps date < 2506, 98 % of the rows
NO_LO = -(2**31)
AGGS3 = [(px.PX_SUM, 0, None), (px.PX_SUM_MUL, 0, 1), (px.PX_COUNT, None, None)]
WIDTH = {"int8": 1, "int32": 4, "int64": 8}


def listed():
    return [
        # A short interactive query, every operator called directly: host work and
        # launch latency are all there is.
        {"name": "scan_20k", "kind": "scan", "rows": 20_011, "parts": 8, "captured": False},
        # The scan-filter-exchange-aggregate query over one ordinary 1M-row batch,
        # replayed from a captured graph as a steady stream of batches is.
        {"name": "scan_1m", "kind": "scan", "rows": 1_000_000, "parts": 8, "captured": True},
        # The same query over a large table: six columns of 1, 4 and 8 bytes go through
        # a selection into the exchange, and few hot groups are aggregated.
        {"name": "scan_30m", "kind": "scan", "rows": 30_000_001, "parts": 64, "captured": False},
        # FilterProject's predicate alone on a large column.
        {"name": "filter_60m", "kind": "filter", "rows": 60_000_000, "dtype": "int32", "keep": 0.3},
        # The exchange alone, with wide rows and many destinations; a ragged row count.
        {"name": "exchange_20m", "kind": "exchange", "rows": 20_000_003, "columns": "wide", "parts": 256},
        # GROUP BY a key whose domain no catalog statistic bounds, ordered by the key.
        {"name": "groupby_hash_10m", "kind": "groupby", "rows": 10_000_019, "groups": 100_000, "dtype": "int64",
         "zipf": False},
        # Filter, join build, join probe and a small group-by on an ordinary batch, as
        # a captured graph.
        {"name": "join_6m", "kind": "join", "rows": 6_000_000, "dim": 200_000, "attrs": 25, "captured": True},
        # The headline chain: exchange of both sides, join per partition, Partial and
        # Final aggregation, skewed keys.
        {"name": "at_scale_60m", "kind": "at_scale", "rows": 60_000_000, "dim": 2_000_000, "parts": 64,
         "attrs": 10_000, "fused": False},
        # The same chain with the probe fused into the Partial aggregation; odd sizes.
        {"name": "at_scale_fused_24m", "kind": "at_scale", "rows": 24_000_007, "dim": 700_003, "parts": 48,
         "attrs": 3_000, "fused": True},
        # A selective join over a wide fact with its payload gathered after the join.
        {"name": "late_20m", "kind": "wide", "rows": 20_000_000, "dim": 1_000_003, "parts": 64, "late": True},
        # A batch as the serving loop forms it at light load: a few fragments, the
        # batch formed from prepared descriptors on every pass.
        {"name": "fragments_served", "kind": "fragments", "count": 6, "scale": 0.25, "sizes": 5, "form": True},
        # The batched fragments workload: 512 fragments, 388M fact rows in all.
        {"name": "fragments_512", "kind": "fragments", "count": 512, "scale": 1.0, "sizes": 4, "form": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["scan", "filter", "exchange", "groupby", "join", "at_scale", "wide", "fragments"])
    if kind == "scan":
        return {"kind": kind, "rows": _log_int(rng, 1e4, 3e7), "parts": rng.choice([1, 3, 8, 64, 200]),
                "captured": rng.random() < 0.5}
    if kind == "filter":
        return {"kind": kind, "rows": _log_int(rng, 1e4, 6e7), "dtype": rng.choice(["int8", "int32", "int64"]),
                "keep": round(rng.choice([0.01, 0.3, 0.98]) * rng.uniform(0.5, 1.0), 3)}
    if kind == "exchange":
        return {"kind": kind, "rows": _log_int(rng, 1e4, 4e7), "columns": rng.choice(["fact", "dim", "wide", "plain"]),
                "parts": _log_int(rng, 2, 1024)}
    if kind == "groupby":
        rows = _log_int(rng, 1e5, 2e7)
        return {"kind": kind, "rows": rows, "groups": _log_int(rng, 100, min(1e6, rows / 4)),
                "dtype": rng.choice(["int32", "int64"]), "zipf": rng.random() < 0.5}
    if kind == "join":
        return {"kind": kind, "rows": _log_int(rng, 1e4, 2e7), "dim": _log_int(rng, 1e3, 2e6),
                "attrs": _log_int(rng, 4, 1000), "captured": rng.random() < 0.5}
    if kind == "at_scale":
        rows, parts = _log_int(rng, 1e6, 5e7), _log_int(rng, 2, 1000)
        return {"kind": kind, "rows": rows, "dim": _log_int(rng, 1e4, 2e6), "parts": parts,
                "attrs": _log_int(rng, 20, min(10_000, 1_000_000 // parts)), "fused": rng.random() < 0.5}
    if kind == "wide":
        return {"kind": kind, "rows": _log_int(rng, 1e6, 4e7), "dim": _log_int(rng, 1e5, 2e6),
                "parts": _log_int(rng, 4, 256), "late": rng.random() < 0.5}
    scale = round(math.exp(rng.uniform(math.log(0.02), 0.0)), 3)
    return {"kind": kind, "count": _log_int(rng, 1, min(512, 256 / scale)), "scale": scale,
            "sizes": rng.randrange(1 << 20), "form": rng.random() < 0.5}


# ------------------------------------------------------------------ inputs ----

class _Draw:
    """Seeded columns on the GPU."""

    def __init__(self, seed):
        self.dev = torch.device("cuda", torch.cuda.current_device())
        self.g = torch.Generator(device=self.dev)
        self.g.manual_seed(int(seed))

    def ints(self, lo, hi, n, dtype=torch.int64):
        """n values uniform in [lo, hi)."""
        return torch.randint(lo, hi, (n,), generator=self.g, device=self.dev, dtype=dtype)

    def perm(self, n):
        return torch.randperm(n, generator=self.g, device=self.dev)

    def zipf(self, nranks, n, s=1.1):
        """n ranks in [0, nranks), P(r) proportional to (r + 1)^-s."""
        cdf = torch.arange(1, nranks + 1, dtype=torch.float64, device=self.dev).pow_(-s).cumsum_(0)
        cdf /= cdf[-1].clone()
        u = torch.rand(n, generator=self.g, device=self.dev, dtype=torch.float64)
        return torch.searchsorted(cdf, u, right=True).clamp_(max=nranks - 1)

    def prices(self, n):
        return self.ints(100, 10**7 + 1, n)

    def amounts(self, n):
        return self.ints(100, 10**6 + 1, n)

    def qtys(self, n):
        return self.ints(1, 51, n)

    def dates(self, n):
        return self.ints(0, DAYS, n, torch.int32)


def _skewed_pair(c, d):
    """A dimension of unique keys 1..dim and a fact whose keys follow Zipf(1.1)."""
    n, nd = c["rows"], c["dim"]
    pk = d.perm(nd) + 1
    attr = d.ints(0, c["attrs"], nd, torch.int32)
    fk = (d.perm(nd) + 1)[d.zipf(nd, n)]
    return {"pk": pk, "attr": attr, "fk": fk, "amount": d.amounts(n), "date": d.dates(n)}


def _fragment_sizes(c):
    """(fact rows, build rows, groups) of each fragment, log-uniform over the batched
    workload's ranges times the case's scale."""
    g = np.random.Generator(np.random.PCG64(c["sizes"]))
    s = c["scale"]

    def log_ints(lo, hi):
        lo, hi = max(1, int(lo)), max(5, int(hi))
        return np.floor(np.exp(g.uniform(np.log(lo), np.log(hi), size=c["count"]))).astype(np.int64)

    return log_ints(1e4 * s, 4e6 * s), log_ints(1e3 * s, 1e6 * s), log_ints(4, 1e5 * s)


# ------------------------------------------------------------------ states ----

def _keep_graph(state):
    """Captures the state's pass once, as a program that repeats it does."""
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        state["pass"]()
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        state["out"] = state["pass"]()
    state["graph"] = graph
    return state


def _zero(*buffers):
    for b in buffers:
        for t in b:
            t.zero_()


def _groups(r):
    return {"keys": r["keys"], "aggs": r["aggs"], "ngroups": r["ngroups"]}


def _scan(c, d):
    n = c["rows"]
    cols = {"key": d.ints(0, 2**20, n), "price": d.prices(n), "qty": d.qtys(n), "date": d.dates(n),
            "flag": d.ints(0, 4, n, torch.int8), "status": d.ints(0, 2, n, torch.int8)}
    p = PlainPipeline(cols, NO_LO, SCAN_HI, nparts=c["parts"])
    _zero([p.sel], p.parts, p.gout)

    def one():
        r = p.run()
        return {"sel": r["sel"], "nsel": r["nsel"], "parts": r["parts"], "offsets": r["offsets"],
                "groups": _groups(r["groups"])}
    state = {"pass": one, "keep": p}
    return _keep_graph(state) if c["captured"] else state


def _join(c, d):
    n, nd = c["rows"], c["dim"]
    cols = {"pk": d.perm(nd) + 1, "attr": d.ints(0, c["attrs"], nd, torch.int32), "fk": d.ints(1, nd + 1, n),
            "amount": d.amounts(n), "date": d.dates(n)}
    p = JoinPipeline(cols, DATE_LO, DATE_HI, max_groups=max(64, c["attrs"]), attr_range=(0, c["attrs"] - 1))
    _zero([p.sel], p.jout, p.gout)

    def one():
        r = p.run()
        return {"sel": r["sel"], "nsel": r["nsel"], "join": r["join"]["cols"], "nout": r["join"]["nout"],
                "groups": _groups(r["groups"])}
    state = {"pass": one, "keep": p}
    return _keep_graph(state) if c["captured"] else state


def _at_scale(c, d):
    p = AtScalePipeline(_skewed_pair(c, d), nparts=c["parts"], nattr_bound=c["attrs"], fused=c["fused"])
    _zero(p.fparts, p.dparts, p.jout, p.pout, p.fout)

    def one():
        r = p.run()
        out = {"dim_offsets": r["dim_offsets"], "fact_offsets": r["fact_offsets"], "fact": p.fparts,
               "dim": p.dparts, "partial": _groups(r["partial"]), "final": _groups(r["final"])}
        if not c["fused"]:
            out["join"] = r["join"]["cols"]
            out["nout"], out["out_seg"] = r["join"]["nout"], r["join"]["out_seg"]
        return out
    return {"pass": one, "keep": p}


def _wide(c, d):
    """The build side is the dimension rows with attr < 1000 of 10000 (about 10 %)."""
    cols = _skewed_pair(dict(c, attrs=10_000), d)
    cols["price"], cols["qty"] = d.prices(c["rows"]), d.qtys(c["rows"])
    keep = cols["attr"] < 1_000
    cols["pk_b"], cols["attr_b"] = cols["pk"][keep], cols["attr"][keep]
    p = WideJoinPipeline(cols, late=c["late"], nparts=c["parts"])
    _zero(p.jout, p.gout if c["late"] else [], p.pout, p.fout)

    def one():
        r = p.run()
        return {"join": r["join"]["cols"], "nout": r["join"]["nout"], "out_seg": r["join"]["out_seg"],
                "payload": p.gout if c["late"] else [], "partial": _groups(r["partial"]),
                "final": _groups(r["final"])}
    return {"pass": one, "keep": p}


def _filter(c, d):
    n, dtype = c["rows"], getattr(torch, c["dtype"])
    # int8: flags and small codes; wider: dates or fixed-point values
    lo, hi = {"int8": (-100, 100), "int32": (0, DAYS), "int64": (-10**9, 10**9)}[c["dtype"]]
    col = d.ints(lo, hi, n, dtype)
    span = max(1, round((hi - lo) * c["keep"]))
    first = lo + (hi - lo - span) // 2
    sel = torch.zeros(n, dtype=torch.int32, device=d.dev)
    nsel = torch.zeros(1, dtype=torch.int64, device=d.dev)
    ws = px.Workspace(px.lib().px_filter_ws_bytes(n))
    return {"pass": lambda: px.px_filter(col, first, first + span, sel=sel, nsel=nsel, ws=ws)}


EXCHANGE_COLS = {"fact": [8, 8, 4], "dim": [8, 4], "wide": [8, 8, 8, 8], "plain": [8, 8, 8, 4, 1, 1]}


def _exchange(c, d):
    n, parts = c["rows"], c["parts"]
    cols = [d.ints(0, 2**20, n)]
    for w in EXCHANGE_COLS[c["columns"]][1:]:
        cols.append({8: d.prices, 4: d.dates, 1: lambda k: d.ints(0, 4, k, torch.int8)}[w](n))
    out = [torch.zeros_like(x) for x in cols]
    offsets = torch.zeros(parts + 1, dtype=torch.int64, device=d.dev)
    ws = px.Workspace(px.lib().px_partition_ws_bytes(n, parts))
    return {"pass": lambda: px.px_partition(cols, 0, parts, out=out, offsets=offsets, ws=ws)}


def _groupby(c, d):
    n, g, dtype = c["rows"], c["groups"], getattr(torch, c["dtype"])
    ids = d.zipf(g, n) if c["zipf"] else d.ints(0, g, n)
    # surrogate keys spread over the type's range: no useful statistic
    names = d.perm(g) * (2**31 // (g + 1)) + d.ints(0, 2**31 // (g + 1), g)
    if dtype == torch.int64:
        names = names * 2**32 + d.ints(0, 2**32, g)
    cols = [names[ids].to(dtype), d.prices(n), d.qtys(n)]
    most = g + g // 4  # the planner's estimate of the group count
    out = [torch.full((most,), torch.iinfo(dtype).max, dtype=dtype, device=d.dev)]
    out += [torch.zeros(most, dtype=torch.int64, device=d.dev) for _ in range(3)]
    ngroups = torch.zeros(1, dtype=torch.int64, device=d.dev)
    ws = px.Workspace(px.lib().px_groupby_ws_bytes(n, most))
    aggs = [(px.PX_SUM, 1, None), (px.PX_SUM_MUL, 1, 2), (px.PX_COUNT, None, None)]

    def one():
        r = px.px_groupby_agg(cols, [0], aggs, max_groups=most, out=out, ngroups=ngroups, ws=ws)
        keys, order = torch.sort(r["keys"][0])  # ORDER BY the key; unused rows hold the largest key
        return {"keys": keys, "aggs": [a[order] for a in r["aggs"]], "ngroups": r["ngroups"]}
    return {"pass": one}


def _fragments(c, d):
    nfact, nbuild, ngroups = _fragment_sizes(c)
    total = int(ngroups.sum())
    # every fragment's results land in its range of shared result columns
    keys = torch.zeros(total, dtype=torch.int32, device=d.dev)
    aggs = [torch.zeros(total, dtype=torch.int64, device=d.dev) for _ in range(3)]
    counts = torch.zeros(len(nfact), dtype=torch.int64, device=d.dev)
    ws, frags, at = px.Workspace(256), [], 0
    for i, (n, nb, ng) in enumerate(zip(nfact.tolist(), nbuild.tolist(), ngroups.tolist())):
        pk, attr = d.perm(nb) + 1, d.ints(0, ng, nb, torch.int32)
        table = px.px_join_build([pk, attr], 0, unique=True, pay_col=1, ws=ws)
        frags.append({"key": d.ints(1, nb + nb // 20 + 1, n), "filter": d.dates(n), "lo": DATE_LO, "hi": DATE_HI,
                      "cols": [d.prices(n), d.qtys(n)], "aggs": AGGS3, "table": table, "group": attr, "group_lo": 0,
                      "group_hi": ng - 1, "max_groups": ng,
                      "out": (keys[at:at + ng], [a[at:at + ng] for a in aggs], counts[i:i + 1])})
        at += ng
    prepared = [px.fragment_descriptor(f) for f in frags]
    state = {"batch": px.FragmentBatch(None, prepared=prepared), "event": None, "prepared": prepared, "frags": frags}

    def one():
        # a batch's plan buffer is in use until its run has completed, so a program
        # runs the batch again only then (other batches may be in flight)
        if state["event"] is not None:
            state["event"].synchronize()
        if c["form"]:
            old = state["batch"]
            state["batch"] = px.FragmentBatch(None, prepared=prepared, ws=old.ws, plan=old.plan)
        state["batch"].run()
        state["event"] = torch.cuda.Event()
        state["event"].record()
        return {"keys": keys, "aggs": aggs, "ngroups": counts}
    state["pass"] = one
    return state


def prepare(case, seed):
    make = {"scan": _scan, "filter": _filter, "exchange": _exchange, "groupby": _groupby, "join": _join,
            "at_scale": _at_scale, "wide": _wide, "fragments": _fragments}[case["kind"]]
    return make(case, _Draw(seed))


def run(state):
    if "graph" in state:
        state["graph"].replay()
        return state["out"]
    return state["pass"]()


def work(case):
    """Bytes of one pass: every input column read once, every output row written once
    (expected row counts where a filter or join decides them)."""
    k, n = case["kind"], case.get("rows", 0)
    if k == "scan":      # six columns in; the selection and the exchanged columns out
        b = 30 * n + SCAN_HI / DAYS * (4 + 30) * n
    elif k == "filter":
        b = WIDTH[case["dtype"]] * n + 4 * case["keep"] * n
    elif k == "exchange":
        b = 2 * sum(EXCHANGE_COLS[case["columns"]]) * n + 8 * case["parts"]
    elif k == "groupby":  # key, price and qty in; a key and three aggregates per group out
        w = WIDTH[case["dtype"]]
        b = (w + 16) * n + (w + 24) * case["groups"]
    elif k == "join":    # fk, amount, date and the dimension in; selection, amount and attr out
        b = 20 * n + 12 * case["dim"] + (DATE_HI - DATE_LO) / DAYS * (4 + 12) * n
    elif k == "at_scale":  # both sides in and exchanged; unfused: the joined amount and attr too
        groups = min(case["dim"], case["parts"] * case["attrs"])
        b = 40 * n + 24 * case["dim"] + (0 if case["fused"] else 12 * n) + 20 * (groups + case["attrs"])
    elif k == "wide":    # the fact's four columns and a tenth of the dimension in
        groups = min(case["dim"] // 10, case["parts"] * 1_000)
        b = 32 * n + 1.2 * case["dim"] + 0.1 * n * 28 + 28 * (groups + 1_000)
    else:                # date, key, price, qty per fact row, the dimension, the groups
        nfact, nbuild, ngroups = (int(x.sum()) for x in _fragment_sizes(case))
        b = 28 * nfact + 12 * nbuild + 28 * min(ngroups, nbuild)
    return {"bytes": float(b), "flops": 0.0}


def exact(case, seed):
    """None: every output is a whole number, equal or wrong."""
    return None
