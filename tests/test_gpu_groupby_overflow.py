"""A group-by whose capacity underestimates the groups: the call reports it, and ends."""
import numpy as np
import pytest
import torch

import oracle
import pxdata
from gpu_helpers import assert_groups_equal, count, dev

pytestmark = pytest.mark.gpu


def _time(f):
    best = 1e9
    for _ in range(4):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        r = f()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best, r


# No statistic (the hash table) and a statistic that no key lies in (the claim table).
@pytest.mark.parametrize("key_range", [None, [(0, 9)]])
@pytest.mark.parametrize("max_groups", [100, 20_000])
def test_many_more_groups_than_capacity(px, key_range, max_groups):
    n = 1_000_000
    g = pxdata.rng(50)
    key = dev(g.permutation(n).astype(np.int64) + 1000)
    val = dev(np.ones(n, np.int64))
    aggs = [(px.PX_SUM, 1, None), (px.PX_COUNT, None, None)]

    def call(mg):
        ws = px.Workspace(px.lib().px_groupby_ws_bytes(n, mg))
        out = [torch.empty(mg, dtype=torch.int64, device="cuda") for _ in range(3)]
        return lambda: px.px_groupby_agg([key, val], [0], aggs, max_groups=mg, key_range=key_range, out=out, ws=ws), ws

    fits, ws = call(n)
    base, r = _time(fits)
    assert count(r["ngroups"]) == n and ws.status() == px.PX_OK
    short, ws = call(max_groups)
    t, r = _time(short)
    print(f"capacity {n}: {base:.3f} ms, {max_groups}: {t:.3f} ms")
    assert ws.status() == px.PX_ERR_CAPACITY
    assert max_groups < count(r["ngroups"]) <= n
    # every row past the capacity walked the whole table: hundreds of times longer
    assert t < 10 * base + 1.0, (t, base)


def test_capacity_short_by_little_reports_every_group(px):
    n, groups = 300_000, 5000
    key = dev((np.arange(n, dtype=np.int64) % groups) * 977 - 10**6)
    aggs = [(px.PX_COUNT, None, None)]
    for key_range in (None, [(10**9, 10**9 + 7)]):
        ws = px.Workspace(1 << 20)
        r = px.px_groupby_agg([key], [0], aggs, max_groups=groups - 1, key_range=key_range, ws=ws)
        assert count(r["ngroups"]) == groups and ws.status() == px.PX_ERR_CAPACITY


def _keys_of_one_bucket(n):
    """n int64 keys whose hashes (MurmurHash3's finalizer of the biased key) agree in their
    low 32 bits: they meet in one place of a table of any size."""
    m1, m2 = pow(0xff51afd7ed558ccd, -1, 2**64), pow(0xc4ceb9fe1a85ec53, -1, 2**64)
    h = (np.arange(1, n + 1, dtype=np.uint64) << np.uint64(32)) | np.uint64(0x1234567)
    for m in (m2, m1):
        h = (h ^ (h >> np.uint64(33))) * np.uint64(m)
    h ^= h >> np.uint64(33)
    return (h ^ np.uint64(1 << 63)).view(np.int64)


@pytest.mark.parametrize("nkeys", [200, 260, 261, 900])
@pytest.mark.parametrize("form", ["plain", "selection", "segments", "stream"])
def test_keys_that_meet_in_one_place(px, nkeys, form):
    """No rows go missing where the keys of a table that is far from full fill more
    neighbouring buckets than a lookup walks."""
    g = pxdata.rng(nkeys)
    n = 40_000
    keys = _keys_of_one_bucket(nkeys)
    if form == "segments":  # two segments need a key narrower than 64 bits; their groups differ in nothing else
        keys = keys.astype(np.int32)
        nkeys = np.unique(keys).size
    k = keys[np.arange(n) % keys.size][g.permutation(n)]
    v = pxdata.random_column(g, n, np.int64)
    aggs = [(px.PX_SUM, 1, None), (px.PX_COUNT, None, None), (px.PX_SUM_MUL, 1, 1)]
    ws = px.Workspace(1 << 20)
    kw = {"max_groups": 2000, "ws": ws}
    pos = np.arange(n)
    if form == "selection":
        pos = np.sort(g.permutation(n)[: n // 2])
        kw.update(sel=dev(pos.astype(np.int32)), nsel=dev(np.array([pos.size])))
    seg = np.array([0, 15_000, n]) if form == "segments" else None
    if seg is not None:
        kw.update(seg=dev(seg))
    ops = [(oracle.SUM, v[pos], None), (oracle.COUNT, None, None), (oracle.SUM_MUL, v[pos], v[pos])]
    if form == "stream":
        out = [torch.empty(2000, dtype=torch.int64, device="cuda") for _ in range(4)]
        ng = torch.zeros(1, dtype=torch.int64, device="cuda")
        for i, (a, b) in enumerate([(0, 300), (300, 20_000), (20_000, 20_000), (20_000, n)]):
            r = px.px_groupby_agg([dev(k[a:b]), dev(v[a:b])], [0], aggs, out=out, ngroups=ng,
                                  flags=px.PX_AGG_STREAM if i == 0 else px.PX_AGG_ACCUMULATE, **kw)
            assert count(ng) == np.unique(k[:b]).size
    else:
        r = px.px_groupby_agg([dev(k), dev(v)], [0], aggs, **kw)
    assert ws.status() == px.PX_OK
    assert_groups_equal(r, oracle.groupby([k[pos]], ops, seg=seg), 1, segmented=seg is not None)


def test_keys_that_meet_in_one_place_over_capacity(px):
    n = 900
    k = dev(_keys_of_one_bucket(n))
    ws = px.Workspace(1 << 20)
    r = px.px_groupby_agg([k], [0], [(px.PX_COUNT, None, None)], max_groups=300, ws=ws)
    assert ws.status() == px.PX_ERR_CAPACITY and 300 < count(r["ngroups"]) <= n
