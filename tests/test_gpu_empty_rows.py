"""Joins whose device row counts are 0 while their buffers have room for many rows: the
kernels that find no row still hold back the next call until the work before is done."""
import numpy as np
import pytest
import torch

import pxdata
from gpu_helpers import count, dev, host

pytestmark = pytest.mark.gpu


def _zero():
    return torch.zeros(1, dtype=torch.int64, device="cuda")


@pytest.mark.parametrize("nsegs", [0, 64])
def test_build_of_no_rows_over_an_earlier_table(px, nsegs):
    n = 300_000
    pk, fk = dev(np.arange(n, dtype=np.int64)), dev(np.arange(n, dtype=np.int64)[::-1])
    seg = dev(np.linspace(0, n, nsegs + 1).astype(np.int64)) if nsegs else None
    noseg = torch.zeros_like(seg) if nsegs else None
    fkseg = seg  # every probe row lies in some segment; the empty table has no row for it
    table = torch.empty(px.lib().px_join_table_bytes(n, nsegs), dtype=torch.uint8, device="cuda")
    ws = px.Workspace(px.lib().px_join_probe_ws_bytes(n))
    for _ in range(5):
        px.px_join_build([pk], 0, seg=seg, table=table, ws=ws)
        px.px_join_build([pk], 0, seg=noseg, d_nrows=_zero(), table=table, ws=ws)
        r = px.px_join_probe(table, [fk], 0, seg=fkseg, build_row=True, ws=ws)
        assert count(r["nout"]) == 0
    assert ws.status() == px.PX_OK


def test_probe_of_no_rows_then_group_by(px):
    g = pxdata.rng(41)
    n, nd = 2_000_000, 50_000
    pk = dev(g.permutation(nd).astype(np.int64))
    fk, amount = dev(g.integers(0, nd, n)), dev(g.integers(0, 100, n))
    attr = dev(g.integers(0, 9, nd).astype(np.int32))
    table = px.px_join_build([pk], 0)
    ws = px.Workspace(max(px.lib().px_join_probe_ws_bytes(n), px.lib().px_groupby_ws_bytes(n, 16)))
    aggs = [(px.PX_SUM, 0, None), (px.PX_COUNT, None, None)]
    for nsel, groups in [(n, 9), (0, 0), (n, 9), (0, 0)]:
        sel = torch.arange(n, dtype=torch.int32, device="cuda")
        r = px.px_join_probe(table, [fk, amount], 0, sel=sel, nsel=dev(np.array([nsel])), carry=[1], payload=[attr],
                             out_seg=True, ws=ws)
        got = px.px_groupby_agg(r["cols"], [1], aggs, max_groups=16, d_nrows=r["nout"], key_range=[(0, 8)], ws=ws)
        assert count(got["ngroups"]) == groups
        assert count(r["nout"]) == nsel and host(r["out_seg"]).tolist() == [0, nsel]
    assert ws.status() == px.PX_OK
