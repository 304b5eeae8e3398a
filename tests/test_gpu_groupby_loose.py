"""GROUP BY without a statistic where the capacity is far above the group count: the table is
used as far as an estimate of the groups says. Parity whatever the estimate does, and a cost
that follows the groups, not the capacity."""
import numpy as np
import pytest
import torch

import oracle
import pxdata
from gpu_helpers import assert_groups_equal, count, dev
from test_gpu_groupby_overflow import _keys_of_one_bucket, _time

pytestmark = pytest.mark.gpu

CAP = 1_200_000  # a table of more than 96 MB with one aggregate or more


def _run(px, keys, n, naggs, **kw):
    """SUM, SUM_MUL, COUNT, .. of keys (one or two columns), against the oracle."""
    g = pxdata.rng(n + naggs)
    a, b = pxdata.random_column(g, n, np.int64), pxdata.random_column(g, n, np.int32)
    at = len(keys)
    aggs = ([(px.PX_SUM, at, None), (px.PX_SUM_MUL, at, at + 1), (px.PX_COUNT, None, None)] * 2)[:naggs]
    pos = kw.pop("pos", np.arange(n))
    ops = ([(oracle.SUM, a[pos], None), (oracle.SUM_MUL, a[pos], b[pos].astype(np.int64)), (oracle.COUNT, None, None)] * 2)[:naggs]
    ws = px.Workspace(1 << 20)
    cap = kw.pop("max_groups", CAP)
    r = px.px_groupby_agg([dev(k) for k in keys] + [dev(a), dev(b)], list(range(at)), aggs, max_groups=cap, ws=ws, **kw)
    assert ws.status() == px.PX_OK
    seg = kw["seg"].cpu().numpy() if "seg" in kw else None
    assert_groups_equal(r, oracle.groupby([k[pos] for k in keys], ops, seg=seg), at, segmented=seg is not None)


# Rows up to 2^20 are read whole by the estimate, more rows by a sample; tiles of 4096.
@pytest.mark.parametrize("n", [1_150_000, 1_300_001])
@pytest.mark.parametrize("groups", [1, 100, 50_000, 10**9])
@pytest.mark.parametrize("naggs", [3, 6])
def test_loose_capacity(px, n, groups, naggs):
    g = pxdata.rng(groups % 977 + n)
    keys = g.integers(-groups, groups, n) if groups > 1 else np.full(n, 7, np.int64)
    _run(px, [keys.astype(np.int64)], n, naggs, max_groups=2 * n if groups == 10**9 else CAP)


def test_loose_capacity_all_rows_read(px):
    n = 1_040_000  # below 2^20 rows; a table of 6 aggregates is large all the same
    _run(px, [pxdata.rng(1).integers(0, 3000, n).astype(np.int64)], n, 6, max_groups=n)


def test_loose_capacity_two_keys_selection_segments_and_row_count(px):
    n = 1_500_000
    g = pxdata.rng(8)
    k0, k1 = g.integers(0, 300, n).astype(np.int32), g.integers(0, 9, n).astype(np.int8)
    pos = np.flatnonzero(g.random(n) < 0.9)
    _run(px, [k0, k1], n, 3, pos=pos, sel=dev(np.concatenate([pos, np.zeros(n - pos.size, np.int64)]).astype(np.int32)),
         nsel=dev(np.array([pos.size])))
    _run(px, [k0, k1], n, 3, seg=dev(np.array([0, 10, 10, 700_000, n])))
    _run(px, [k0, k1], n, 3, pos=np.arange(5000), d_nrows=dev(np.array([5000])))
    _run(px, [k0, k1], n, 3, pos=np.arange(0), d_nrows=dev(np.array([0])))


@pytest.mark.parametrize("naggs", [3, 6])
def test_an_estimate_that_is_far_too_low(px, naggs):
    """Keys whose hashes look like few: every register of the estimate stays at its lowest
    value. The table that it asks for cannot hold them."""
    n = 1_200_000
    h = (np.arange(n, dtype=np.uint64) * np.uint64(0x9e3779b97f4a7c15)) | np.uint64(1 << 52)
    m1, m2 = pow(0xff51afd7ed558ccd, -1, 2**64), pow(0xc4ceb9fe1a85ec53, -1, 2**64)
    for m in (m2, m1):
        h = (h ^ (h >> np.uint64(33))) * np.uint64(m)
    h ^= h >> np.uint64(33)
    keys = (h ^ np.uint64(1 << 63)).view(np.int64)
    keys[5] = np.int64(2**63 - 1)  # the code that reads as an empty slot
    _run(px, [keys], n, naggs)


def test_keys_that_meet_in_one_place_of_a_loose_table(px):
    n = 1_100_000
    _run(px, [np.resize(_keys_of_one_bucket(900), n)], n, 3)


def test_loose_capacity_costs_little(px):
    n = 4_000_000
    for groups in (100, 100_000):
        g = pxdata.rng(groups)
        key = dev(g.integers(0, groups, n) * 10**9)
        val = dev(np.ones(n, np.int64))
        aggs = [(px.PX_SUM, 1, None), (px.PX_SUM_MUL, 1, 1), (px.PX_COUNT, None, None)]
        us = {}
        for cap in (groups + groups // 4, n):
            ws = px.Workspace(px.lib().px_groupby_ws_bytes(n, cap))
            out = [torch.empty(cap, dtype=torch.int64, device="cuda") for _ in range(4)]
            us[cap], r = _time(lambda: px.px_groupby_agg([key, val], [0], aggs, max_groups=cap, out=out, ws=ws))
            assert count(r["ngroups"]) == groups
        # the whole table cleared and scanned took 3 to 5 times as long
        assert us[n] < 1.7 * us[groups + groups // 4], us


def test_codes_that_the_sample_does_not_see(px):
    """One key in all rows but a stretch of distinct ones between two tiles that the estimate
    reads: they find room, without the rows being gone through by one block (100 ms)."""
    def read(t):  # the tile of the t-th eight that is read: MurmurHash3's finalizer of t
        h, m = t, 2**64 - 1
        h = (h ^ h >> 33) * 0xff51afd7ed558ccd & m
        h = (h ^ h >> 33) * 0xc4ceb9fe1a85ec53 & m
        return t * 8 + (h ^ h >> 33) % 8

    tile, n = 4096, 6_000_000
    gaps = [(read(t + 1) - read(t) - 1, read(t) + 1) for t in range(n // tile // 8 - 1)]
    tiles, first = max(gaps)
    assert tiles >= 9
    us = {}
    for burst in (False, True):
        key = np.full(n, 5, np.int64)
        if burst:
            key[first * tile:(first + tiles) * tile] = 1000 + np.arange(tiles * tile)
        val = np.arange(n, dtype=np.int64)
        ws = px.Workspace(px.lib().px_groupby_ws_bytes(n, n))
        out = [torch.empty(n, dtype=torch.int64, device="cuda") for _ in range(3)]
        cols = [dev(key), dev(val)]
        us[burst], r = _time(lambda: px.px_groupby_agg(cols, [0], [(px.PX_SUM, 1, None), (px.PX_COUNT, None, None)],
                                                       max_groups=n, out=out, ws=ws))
        assert ws.status() == px.PX_OK
        assert_groups_equal(r, oracle.groupby([key], [(oracle.SUM, val, None), (oracle.COUNT, None, None)]), 1)
    assert us[True] < 3 * us[False] + 0.1, us
