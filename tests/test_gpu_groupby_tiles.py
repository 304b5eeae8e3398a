"""GROUP BY without a statistic at the edges of its tiles: 2048 rows of a block, 512 of them
at a time."""
import numpy as np
import pytest

import oracle
import pxdata
from gpu_helpers import assert_groups_equal, dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [511, 512, 513, 2047, 2048, 2049, 4095, 4096, 4097, 304 * 2048 - 1, 304 * 2048 + 1])
@pytest.mark.parametrize("groups", [3, 10**6])
def test_rows_around_a_tile(px, n, groups):
    g = pxdata.rng(n)
    k, v = g.integers(0, groups, n), pxdata.random_column(g, n, np.int64)
    ws = px.Workspace(1 << 20)
    r = px.px_groupby_agg([dev(k), dev(v)], [0], [(px.PX_SUM, 1, None), (px.PX_COUNT, None, None)], max_groups=n, ws=ws)
    assert ws.status() == px.PX_OK
    assert_groups_equal(r, oracle.groupby([k], [(oracle.SUM, v, None), (oracle.COUNT, None, None)]), 1)
