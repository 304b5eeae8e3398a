"""px_partition where a block's shared memory is just below or above 48 KB, the size up
to which a kernel needs no leave for more, and at one block per SM. Each call runs in a
process of its own: an earlier call that took more of the same kernel would have raised
its limit already."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = """
import json, sys
import numpy as np
import torch
import oracle, pxdata
import paper_2606_24647_gb300 as px
n, nparts, widths, config = json.loads(sys.argv[1])
g = pxdata.rng(n + nparts)
types = {8: np.int64, 4: np.int32, 1: np.int8}
cols = [pxdata.random_column(g, n, types[w]) for w in widths]
for c in config:
    out, off = px.px_partition([torch.from_numpy(x).cuda() for x in cols], 0, nparts, 3,
                               config=None if c is None else tuple(c))
    want, woff = oracle.partition(cols, 0, nparts, 3)
    np.testing.assert_array_equal(off.cpu().numpy(), woff)
    for a, b in zip(out, want):
        np.testing.assert_array_equal(a.cpu().numpy()[:n], b)
print("same")
"""


@pytest.mark.parametrize("n,nparts,widths,config", [
    (5000, 1023, [8, 4], [None]),                    # rows held in registers, tiles of 1024 rows
    (700_001, 681, [8, 4], [None]),                  # the same, tiles of 2048
    (60_001, 55, [8, 1, 1], [None]),                 # staged tiles of 2048
    (60_001, 27, [8, 8, 8, 8, 1, 1], [None]),        # staged tiles of 1024
    (60_001, 64, [8, 8, 4], [[8, 1], [4, 1], [2, 1], [0, 1]]),  # one block per SM
    (60_001, 200, [8, 8, 4], [[0, 1]]),
])
def test_partition_at_shared_memory_limits(px, n, nparts, widths, config):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD, json.dumps([n, nparts, widths, config])], cwd=root,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.split() == ["same"], r.stdout + r.stderr
