"""Items of the fused path around the counts at which their candidates turn from a warp
each to bands of rows, spots and lone pixels apart, and bright areas that fill more than
a band's list, against the oracle: plateaus, ties, panel edges, NaN."""
import numpy as np
import pytest

import paper_2206_11297_gb300 as rb
from gpu_util import FUSED_DENSE, assert_parity

pytestmark = pytest.mark.gpu

GEOM = (2, 61, 96)  # one item; ten candidates a band make 80 (eight panels of one band)
LOOSE = dict(amax_thr=200.0, atot_thr=300.0, npix_min=1, npix_max=400, son_min=1.0, max_peaks=8192)


def background(seed):
    return np.random.default_rng(seed).normal(10.0, 3.0, (2, *GEOM)).astype(np.float32)


@pytest.mark.parametrize("path", [rb.PATH_FUSED, FUSED_DENSE])
@pytest.mark.parametrize("rank", [1, 3])
@pytest.mark.parametrize("count", [79, 80, 81, 160, 256, 257, 400, 900])
def test_lone_pixels_and_clusters(count, rank, path):
    rng = np.random.default_rng([count, rank])
    f = background([1, count])
    lone = rng.choice(f[0].size, count, replace=False)
    f[0].reshape(-1)[lone] = rng.choice([500.0, 800.0, 3000.0], count).astype(np.float32)
    # clusters of six, equal and falling, over row ends too
    seeds = rng.choice(f[1].size - 200, max(1, count // 6), replace=False)
    for k, v in enumerate((900.0, 900.0, 700.0, 500.0, 900.0, 400.0)):
        f[1].reshape(-1)[seeds + (0, 1, 2, 96, 97, 98)[k]] = v
    f[1].reshape(-1)[::977] = np.nan
    assert_parity(f, rb.default_params(rank=rank, **LOOSE), path, check_decompress=False)


@pytest.mark.parametrize("path", [rb.PATH_FUSED, FUSED_DENSE])
@pytest.mark.parametrize("change", [{}, dict(rank=1), dict(rank=5, ring_r0=7), dict(rank=7, ring_r0=9, ring_dr=4)])
@pytest.mark.parametrize("rows", [4, 5, 6, 12, 61])
def test_bright_areas(rows, change, path):
    # `rows` bright rows of 96 pixels: 384 and 480 fit a list of 512, 576 do not
    f = background([2, rows])
    y, x = np.mgrid[:rows, :96]
    f[0, 0, :rows] += (600.0 + 40.0 * np.sin(0.3 * x) * np.cos(0.4 * y)).astype(np.float32)
    f[0, 1, 61 - rows:] = 750.0  # a plateau: only its first pixel can be a maximum
    f[1, :, :rows] += 500.0
    f[1, 1, ::7, ::5] = 4000.0
    f[1, 0, 1, 3::31] = np.nan
    assert_parity(f, rb.default_params(**{**LOOSE, **change}), path, check_decompress=False)
