"""The length-table update on runs of rays that share a cell, broken by misses and
by warp, tile and grid edges, against the oracle's table.  Integers: exact."""
import numpy as np
import pytest
import torch

import oracle
from paper_2506_11273_gb300 import rr
from paper_2506_11273_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("run", [1, 3, 32, 100])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 255, 257, 8 * 152 * 256 + 33])
def test_runs_match_oracle(n, run):
    lo, hi = np.zeros(3, np.float32), np.full(3, 2.0, np.float32)
    base = W.random_rays_in_box(-(-n // run), [-0.1] * 3, [2.1] * 3, seed=n + run)
    rays = base.subset(np.repeat(np.arange(len(base)), run)[:n])
    rng = W.rng_for(n * 7 + run)
    hits = np.zeros((n, 4), np.float32)
    hits[:, 0] = rng.choice(np.array([1e-6, 0.3, 1.0, 5.0, 1e3, 1e30, 0.0], np.float32), n)  # clamped at both ends
    tri = rng.integers(0, 1000, n).astype(np.uint32)
    miss = rng.random(n) < 0.1
    tri[miss] = W.MISS
    hits[miss, 0] = np.inf
    hits[:, 3] = tri.view(np.float32)
    o, d, _ = rr.to_device_rays(rays)
    table = rr.LengthTable(lo, hi)
    want = oracle.LengthTable(oracle.largest_extent(lo, hi))
    for _ in range(2):
        table.accumulate(o, d, torch.from_numpy(hits).cuda())
        want.accumulate(lo, hi, rays.o_tmin, rays.d_tmax, hits)
    s, c = table.read()
    assert np.array_equal(s, want.sum) and np.array_equal(c, want.cnt)
    table.close()
