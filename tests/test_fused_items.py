"""The fused path's work items at the sizes where they can go wrong, against the
oracle: panels cut into row bands (small batches) and whole (large ones), and
chunks whose non-zero residuals are listed, up to and past the list's limits."""
import numpy as np
import pytest

import oracle
import paper_2206_11297_gb300 as rb
from gpu_util import FUSED_DENSE, assert_parity, gpu_compress, oparams
from synthetic import FrameRecipe, make_frame

pytestmark = pytest.mark.gpu


def frames_of(geom, n, seed):
    r = FrameRecipe(geom, peaks=("uniform", 2, 12), seed=seed)
    return np.stack([make_frame(r, k) for k in range(n)])


@pytest.mark.parametrize("path", [rb.PATH_FUSED, FUSED_DENSE])
@pytest.mark.parametrize("geom", [(3, 41, 52), (2, 8, 388), (1, 185, 388), (1, 67, 1024), (5, 1, 4)])
@pytest.mark.parametrize("change", [{}, dict(lorenzo_dims=3), dict(abs_eb=0.05, quant_radius=8)])
def test_bands_of_small_batches(geom, path, change):
    f = frames_of(geom, 2, seed=sum(geom))
    f[1].reshape(-1)[::7] = 1e30      # prequantisation outliers, more than an item lists
    f[1].reshape(-1)[3::1013] = np.nan
    assert_parity(f, rb.default_params(atot_thr=300.0, **change), path, check_decompress=False)


def test_batch_size_does_not_change_a_frame():
    # 1 frame: many bands; 300: fewer; 2,600 one-item frames: whole panels
    geom, params = (3, 41, 52), rb.default_params(atot_thr=300.0)
    few = frames_of(geom, 4, seed=3)
    few[2].reshape(-1)[::50] = 1e30
    want = [oracle.compress_frame(x, oparams(params))[1] for x in few]
    for n in (1, 300, 2600):
        f = np.tile(few, (-(-n // 4), 1, 1, 1))[:n]
        st, nb, streams = gpu_compress(f, params, path=rb.PATH_FUSED)
        assert (st == 0).all()
        assert all(np.array_equal(streams[k], want[k % 4]) for k in range(n))


def frame_with(residuals):
    """A one-panel frame whose 2-D Lorenzo residuals at eb 10 and 2 x 2 bins are these."""
    q = np.cumsum(np.cumsum(residuals, axis=0), axis=1)
    return (20.0 * q).astype(np.float32).repeat(2, axis=0).repeat(2, axis=1)[None]


@pytest.mark.parametrize("others", [0, 1, 31, 32, 33, 511, 512, 513])
@pytest.mark.parametrize("last", [4, 4092, 4096])
@pytest.mark.parametrize("kind", ["ones", "outliers", "escapes"])
def test_listed_chunks(others, last, kind):
    # two full chunks and one of `last` symbols; `others` non-zero residuals in the second
    cols = 4
    n = 2 * 4096 + last
    d = np.zeros(n, np.int64)
    rng = np.random.default_rng([others, last])
    at = 4096 + rng.choice(4096, others, replace=False)
    value = {"ones": [1], "outliers": [600, 1], "escapes": [200, -300, 2]}[kind]
    # every step is taken back in the same column, so that the values stay exact
    d[at] = np.resize(value, others) * np.resize([1, -1], others)
    d[5], d[n - 1] = 1, -1
    f = frame_with(d.reshape(n // cols, cols))
    assert np.abs(f).max() < 2 ** 24
    params = rb.default_params(amax_thr=1e30, max_peaks=0)
    assert_parity(f[None], params, rb.PATH_FUSED, check_decompress=False)


@pytest.mark.parametrize("path", [rb.PATH_FUSED, rb.PATH_PLAIN])
@pytest.mark.parametrize("geom", [(70, 9, 36), (33, 4, 8), (3, 2, 1736)])
def test_panel_stacks(geom, path):
    # more panels than a stack item holds at once; slices cut inside a panel
    f = frames_of(geom, 2, seed=sum(geom))
    f[0].reshape(-1)[::11] = 4000.0   # outliers and escapes on both sides of a slice
    assert_parity(f, rb.default_params(atot_thr=300.0, lorenzo_dims=3, abs_eb=1.0, max_peaks=8192), path)


@pytest.mark.parametrize("geom,bin_w", [((3, 5, 8200), 2), ((4, 6, 27), 2), ((2, 7, 30), 3)])
def test_stack_decompression_of_odd_and_wide_rows(geom, bin_w):
    f = frames_of(geom, 2, seed=sum(geom))
    f[1].reshape(-1)[::97] = 1e30
    assert_parity(f, rb.default_params(atot_thr=300.0, lorenzo_dims=3, bin_w=bin_w), rb.PATH_PLAIN)
