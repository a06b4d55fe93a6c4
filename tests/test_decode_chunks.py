"""The chunk decoder (a warp per 4,096-symbol chunk, its lanes starting at
guessed bits) on codes and sizes where it can go wrong, against the oracle:
chunks that end inside a lane's range, words beyond the shared-memory stage,
codes past the 12-bit prefix table, one-symbol codes, long runs."""
import numpy as np
import pytest

import oracle
import paper_2206_11297_gb300 as rb
from gpu_util import dec_paths, gpu_decompress, oparams

pytestmark = pytest.mark.gpu


def residuals(kind, m, rng):
    if kind == "one":
        return np.zeros(m, np.int64)
    if kind == "runs":  # a length-1 code with a few others: the sparse lists
        return np.where(rng.random(m) < 0.02, rng.integers(-3, 4, m), 0)
    if kind == "bursts":  # around and past the eight listed symbols a lane keeps of its range
        dense = (np.arange(m) // 96) % 4 == 0
        return np.where(rng.random(m) < np.where(dense, 0.12, 0.005), rng.integers(-3, 4, m), 0)
    if kind == "crowded":  # a length-1 code, more than 1,024 other symbols per chunk
        return np.where(rng.random(m) < 0.45, rng.integers(-2, 3, m), 0)
    if kind == "flat":  # ten bits a symbol: more words than the stage holds
        return rng.integers(-511, 512, m)
    if kind == "fib":  # Fibonacci counts: the longest codes
        counts, a, b = [], 1, 1
        while sum(counts) + a < m:
            counts.append(a)
            a, b = b, a + b
        sym = np.repeat(np.arange(len(counts)), counts)
        sym = np.concatenate([sym, np.full(m - len(sym), len(counts) - 1)]) if counts else np.zeros(m, np.int64)
        return rng.permutation(sym) - 5
    if kind == "outliers":  # code 0 is common
        return np.where(rng.random(m) < 0.3, rng.choice([-600, 700, 5000], m), rng.integers(-2, 3, m))
    raise ValueError(kind)


@pytest.mark.parametrize("kind", ["one", "runs", "bursts", "crowded", "flat", "fib", "outliers"])
@pytest.mark.parametrize("panels,width", [(1, 1), (1, 33), (3, 1365), (1, 4096), (2, 2049), (5, 4093)])
def test_chunk_decoder(kind, panels, width):
    rng = np.random.default_rng([len(kind), panels, width])
    # one-row panels at bin 1x1: the residual of a bin is its step from the bin before
    d = residuals(kind, panels * width, rng).reshape(panels, 1, width)
    frame = (20.0 * np.cumsum(d, axis=2)).astype(np.float32)
    params = rb.default_params(bin_h=1, bin_w=1, amax_thr=1e30, max_peaks=0)
    st, ref = oracle.compress_frame(frame, oparams(params))
    assert st == 0
    st, want = oracle.decompress_frame(ref, frame.shape)
    assert st == 0
    for path in dec_paths(frame.shape, params):
        rec, status = gpu_decompress([ref, ref], frame.shape, params, dec_path=path)
        assert (status == 0).all()
        for k in range(2):
            assert np.array_equal(rec[k].view(np.uint32), want.view(np.uint32))
        # a chunk index that gives the first chunk a word more than it uses is refused
        off = oracle.section_offsets(oracle.parse_header(ref))
        if panels * width > 4096:
            bad = ref.copy()
            bad[off["chunk_index"]:off["chunk_index"] + 8].view(np.uint32)[1] += 1
            _, status = gpu_decompress([bad], frame.shape, params, dec_path=path)
            assert status[0] == rb.ERR_CORRUPT_STREAM
