"""Streams of group-by calls without a statistic: each group keeps its output row, small
calls write out only what they touch, and their cost does not follow the capacity."""
import numpy as np
import pytest
import torch

import oracle
import pxdata
from gpu_helpers import assert_groups_equal, count, dev, host
from test_gpu_groupby_overflow import _time

pytestmark = pytest.mark.gpu


class _Stream:
    def __init__(self, px, aggs, max_groups, key_dtype=torch.int64):
        self.px, self.aggs, self.cap, self.first = px, aggs, max_groups, True
        self.ws = px.Workspace(1 << 20)
        self.out = [torch.empty(max_groups, dtype=key_dtype, device="cuda")] + \
                   [torch.empty(max_groups, dtype=torch.int64, device="cuda") for _ in aggs]
        self.ng = torch.zeros(1, dtype=torch.int64, device="cuda")

    def feed(self, cols, **kw):
        self.res = self.px.px_groupby_agg(
            cols, [0], self.aggs, max_groups=self.cap, out=self.out, ws=self.ws, ngroups=self.ng,
            flags=self.px.PX_AGG_STREAM if self.first else self.px.PX_AGG_ACCUMULATE, **kw)
        self.first = False


# rows of the calls: below an eighth of a large table's slots (2.25 per group or 1.45, more
# than 2^19) a call writes out the groups that it touches, else all
CALLS = [3, 0, 40_000, 1, 700, 2000, 130_000, 31, 0, 1023, 1024, 1025]


@pytest.mark.parametrize("naggs", [0, 2, 3, 6])
@pytest.mark.parametrize("ngroups,cap", [(1, 1), (900, 1000), (60_000, 60_100), (100_000, 400_000)])
def test_stream_of_small_and_large_calls(px, naggs, ngroups, cap):
    g = pxdata.rng(ngroups + naggs)
    names = g.integers(-2**62, 2**62, ngroups)
    names[0] = 2**63 - 1  # the code that reads as an empty slot
    n = sum(CALLS)
    k = names[g.integers(0, ngroups, n)]
    a, b = pxdata.random_column(g, n, np.int64), pxdata.random_column(g, n, np.int32)
    aggs = ([(px.PX_SUM, 1, None), (px.PX_COUNT, None, None), (px.PX_SUM_MUL, 1, 2)] * 2)[:naggs]
    s = _Stream(px, aggs, cap)
    at, rows = 0, {}
    for c in CALLS:
        kw = {"d_nrows": dev(np.array([c]))} if c else {}
        pad = 5 if c else 0  # capacity beyond the device row count
        part = slice(at, at + c)
        cols = [dev(np.concatenate([x[part], x[:pad]])) for x in (k, a, b)]
        s.feed(cols, **kw)
        at += c
        ng = count(s.ng)
        keys = host(s.out[0], ng)
        assert ng == np.unique(k[:at]).size == np.unique(keys).size
        for row, key in enumerate(keys.tolist()):
            assert rows.setdefault(key, row) == row  # a group's row stays
    assert s.ws.status() == px.PX_OK
    av, bv = a, b.astype(np.int64)
    ops = ([(oracle.SUM, av, None), (oracle.COUNT, None, None), (oracle.SUM_MUL, av, bv)] * 2)[:naggs]
    assert_groups_equal(s.res, oracle.groupby([k], ops), 1)


def test_stream_with_segments_and_selection(px):
    g = pxdata.rng(5)
    s = _Stream(px, [(px.PX_SUM, 1, None)], 50_000, torch.int32)
    oseg = torch.empty(50_000, dtype=torch.int32, device="cuda")
    ks, vs, segs = [], [], []
    for n in (500, 30_000, 800):
        k, v = g.integers(0, 700, n).astype(np.int32), g.integers(-9, 9, n)
        pos = np.flatnonzero(g.random(n) < 0.8)
        seg = np.array([0, pos.size // 3, pos.size])
        sel = np.concatenate([pos, np.zeros(n - pos.size, np.int64)]).astype(np.int32)
        s.feed([dev(k), dev(v)], sel=dev(sel), nsel=dev(np.array([pos.size])), seg=dev(seg), out_seg=oseg)
        ks.append(k[pos]); vs.append(v[pos]); segs.append(np.repeat([0, 1], np.diff(seg)))
    k, v, q = (np.concatenate(x) for x in (ks, vs, segs))
    o = np.argsort(q, kind="stable")
    want = oracle.groupby([k[o]], [(oracle.SUM, v[o], None)], seg=np.array([0, (q == 0).sum(), q.size]))
    assert s.ws.status() == px.PX_OK
    assert_groups_equal(s.res, want, 1, segmented=True)


def test_stream_over_capacity(px):
    s = _Stream(px, [(px.PX_COUNT, None, None)], 100)
    for i, n in enumerate((50, 50, 50, 3000)):
        s.feed([dev(np.arange(i * 50, i * 50 + n, dtype=np.int64))])
        assert count(s.ng) == i * 50 + n
        assert s.ws.status() == (px.PX_OK if i < 2 else px.PX_ERR_CAPACITY)
    assert np.unique(host(s.out[0], 100)).size == 100 and (host(s.out[1], 100) >= 1).all()


def test_small_calls_do_not_pay_for_the_capacity(px):
    g = pxdata.rng(6)
    names = g.integers(-2**62, 2**62, 100_000)
    us = {}
    for cap in (125_000, 10_000_000):
        s = _Stream(px, [(px.PX_SUM, 1, None), (px.PX_SUM_MUL, 1, 1), (px.PX_COUNT, None, None)], cap)
        s.feed([dev(names), dev(names)])
        part = names[g.integers(0, names.size, 10_000)]
        batch = [dev(part), dev(part)]
        us[cap], _ = _time(lambda: s.feed(batch))
        assert count(s.ng) == np.unique(names).size
    # every slot scanned and every group written out took more than three times as long
    assert us[10_000_000] < 2 * us[125_000], us
