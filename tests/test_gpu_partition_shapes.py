"""Launch shapes of the exchange through a selection: every one gives the oracle's result."""
import numpy as np
import pytest

import oracle
import pxdata
from gpu_helpers import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("types", [[np.int64, np.int64, np.int32], [np.int64] * 3 + [np.int32, np.int8, np.int8]])
@pytest.mark.parametrize("nparts", [1, 8, 64, 1000])
def test_shapes_through_a_selection(px, types, nparts):
    g = pxdata.rng(nparts)
    n = 30_011
    cols = [pxdata.random_column(g, n, t) for t in types]
    sel = np.flatnonzero(g.random(n) < 0.9).astype(np.int32)
    want, woff = oracle.partition(cols, 0, nparts, 1, sel=sel)
    for items in (0, 2, 4, 8):
        for blocks in (0, 1, 2, 3):
            out, off = px.px_partition([dev(c) for c in cols], 0, nparts, 1, sel=dev(sel), nsel=dev(np.array([sel.size])),
                                       config=(items, blocks))
            np.testing.assert_array_equal(host(off), woff)
            for a, b in zip(out, want):
                np.testing.assert_array_equal(host(a, sel.size), b)
