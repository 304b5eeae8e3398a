"""Fused fragments with skewed keys: parity around the line between block accumulators in
shared memory and reductions into the global arrays, and no cliff below it."""
import numpy as np
import pytest
import torch

import oracle
import pxdata
from gpu_helpers import dev
from test_gpu_fragments import _check

pytestmark = pytest.mark.gpu


def _fragment(px, seed, n, nb, ngroups, naggs):
    """Zipf(1.1) join keys; the hottest keys' groups are hot too."""
    g = pxdata.rng(seed)
    pk = (g.permutation(nb) + 1).astype(np.int64)
    attr = g.integers(0, ngroups, nb).astype(np.int32)
    key = pk[pxdata.zipf_ranks(g, nb, n, 1.1) - 1]
    a, b = pxdata.random_column(g, n, np.int64), pxdata.random_column(g, n, np.int64)
    date = g.integers(0, 100, n).astype(np.int32)
    aggs = [(px.PX_COUNT, None, None), (px.PX_SUM, 0, None), (px.PX_SUM_MUL, 0, 1), (px.PX_SUM, 1, None)][:naggs]
    d_attr = dev(attr)
    f = {"key": dev(key), "filter": dev(date), "lo": 0, "hi": 60, "cols": [dev(a), dev(b)], "aggs": aggs,
         "table": px.px_join_build([dev(pk), d_attr], 0, unique=True, pay_col=1), "group": d_attr, "group_lo": 0,
         "group_hi": ngroups - 1, "max_groups": ngroups}
    pr, br, _ = oracle.join(pk, key, sel=oracle.filter(date, 0, 60))
    ops = [(oracle.COUNT, None, None), (oracle.SUM, a[pr], None), (oracle.SUM_MUL, a[pr], b[pr]), (oracle.SUM, b[pr], None)]
    return f, oracle.groupby([attr[br]], ops[:naggs])


# 8 bytes per group and aggregate: 42 KB hold 1792 groups of three, 1344 of four, 2688 of two
@pytest.mark.parametrize("naggs,ngroups", [(3, 500), (3, 1025), (3, 1792), (3, 1793), (3, 4000), (4, 1344), (4, 1345),
                                           (2, 2688), (2, 2689)])
def test_skewed_fragments_equal_the_oracle(px, naggs, ngroups):
    f, want = _fragment(px, 70 + ngroups, 60_007, 20_011, ngroups, naggs)
    fb = px.FragmentBatch([f])
    res = fb.run()[0]
    torch.cuda.synchronize()
    assert fb.ws.status() == px.PX_OK
    _check(res, want, naggs)


def test_skewed_fragments_of_a_few_more_groups_take_no_longer(px):
    """1100 hot and cold groups against 1000: a step from shared accumulators to reductions
    at one address would double the time (405 and 950 us measured on 48M rows)."""
    us = {}
    for ngroups in (1000, 1100):
        batch = []
        for i in range(4):
            f, _ = _fragment(px, 90 + i, 20_000, 500_000, ngroups, 3)
            n = 3_000_000  # the rows repeated: only the time matters
            rep = lambda t: t.repeat(n // t.numel() + 1)[:n].contiguous()
            batch.append(dict(f, key=rep(f["key"]), filter=rep(f["filter"]), cols=[rep(c) for c in f["cols"]]))
        fb = px.FragmentBatch(batch)
        times = []
        for _ in range(9):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            fb.run()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        us[ngroups] = min(times)
    assert us[1100] < 1.6 * us[1000], us
