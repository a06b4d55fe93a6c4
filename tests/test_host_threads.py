"""Contexts of their own on two host threads and streams: each thread's calls go
through, whatever shared memory the other's kernels take, and write its bytes."""
import threading

import numpy as np
import pytest

import paper_2206_11297_gb300 as rb
from synthetic import FrameRecipe, make_frame

pytestmark = pytest.mark.gpu


def make(case, large):
    """(geometry, parameters, path, dense variant): two contexts whose launches of one
    kernel take different amounts of shared memory."""
    if case == "dense":
        return (3, 41, 52), rb.default_params(atot_thr=300.0), rb.PATH_FUSED, large
    if case == "wide":
        return (1, 4, 16000 if large else 12000), rb.default_params(atot_thr=300.0), rb.PATH_PLAIN, False
    side = 63 if large else 41
    return (2, 40, 44), rb.default_params(atot_thr=300.0, roi_coder=1, roi_h=side, roi_w=side), rb.PATH_PLAIN, False


@pytest.mark.parametrize("case", ["dense", "wide", "windows"])
def test_two_threads_launch_beside_each_other(case):
    import torch
    errors, outputs, start = [], {}, threading.Barrier(2)

    def work(large):
        try:
            geom, params, path, dense = make(case, large)
            r = FrameRecipe(geom, peaks=("fixed", 4), seed=5)
            frames = torch.from_numpy(np.stack([make_frame(r, k) for k in range(2)])).cuda()
            with rb.Context(geom, params, max_frames=2) as ctx:
                ctx.set_path(path)
                if dense:
                    ctx.set_fused_dense_peaks(True)
                stream = torch.cuda.Stream()
                first = ctx.compress(frames)
                torch.cuda.synchronize()
                want = [t.clone() for t in first]
                torch.cuda.synchronize()
                start.wait(60)
                for _ in range(3000):
                    ctx.compress(frames, out=first[0], frame_bytes=first[1], status=first[2],
                                 out_stride=first[0].shape[1], stream=stream)
                stream.synchronize()
                outputs[large] = [t.cpu().numpy() for t in (*first, *want)]
        except Exception as e:  # reported by the test's thread
            errors.append(f"{case}, large={large}: {e}")
            start.abort()

    threads = [threading.Thread(target=work, args=(large,)) for large in (False, True)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for out, nb, st, out0, nb0, st0 in outputs.values():
        assert (st == rb.OK).all() and np.array_equal(st, st0) and np.array_equal(nb, nb0)
        assert all(np.array_equal(out[k, :nb[k]], out0[k, :nb[k]]) for k in range(2))
