"""The plain path's peak stage around the number of listed pixels at which it
turns from a warp per pixel to the local-maximum rule a thread per pixel, with
ties, plateaus, panel edges and NaN, against the oracle."""
import numpy as np
import pytest

import paper_2206_11297_gb300 as rb
from gpu_util import assert_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hot", [1, 127, 128, 129, 257, 1500, 4096, 4097, 6000])
@pytest.mark.parametrize("rank", [1, 3])
def test_listed_pixels(hot, rank):
    rng = np.random.default_rng([hot, rank])
    f = rng.normal(10.0, 3.0, (2, 2, 61, 97)).astype(np.float32)
    for k, frame in enumerate(f):
        # clusters of equal and falling values, some at the panels' edges
        seeds = rng.choice(frame.size, max(1, hot // 6), replace=False)
        at = np.unique(np.concatenate([seeds, seeds + 1, seeds + 97, seeds + 98, seeds + 2, seeds - 97]))
        at = rng.permutation(at[(at >= 0) & (at < frame.size)])
        more = np.setdiff1d(np.arange(frame.size), at)
        at = np.concatenate([at, rng.choice(more, hot, replace=False)])[:hot]
        frame.reshape(-1)[at] = rng.choice([500.0, 800.0, 800.0, 3000.0], hot).astype(np.float32)
        if k:
            frame.reshape(-1)[::211] = np.nan
    params = rb.default_params(rank=rank, amax_thr=200.0, atot_thr=300.0, npix_min=1, son_min=1.0, max_peaks=8192)
    assert_parity(f, params, rb.PATH_PLAIN, check_decompress=False)
