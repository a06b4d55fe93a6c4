"""The 3-D predictor's stack items when their bounded waits run out (the context's
poll limit is 0 or too small: nothing spins for long, nothing faults): each frame
reports ROIBIN_ERR_TIMEOUT or the oracle's bytes, and the next call at the default
limit writes the oracle's bytes whatever the calls before it left unfinished."""
import numpy as np
import pytest

import oracle
import paper_2206_11297_gb300 as rb
from gpu_util import oparams
from synthetic import FrameRecipe, make_frame

pytestmark = pytest.mark.gpu

GEOM = (4, 120, 256)  # nine stack items a frame
LIMITS = [0, 1, 3, 10, 30, 60, 100, 300]


def frames_of(n, seed):
    r = FrameRecipe(GEOM, peaks=("uniform", 2, 12), seed=seed)
    return np.stack([make_frame(r, k) for k in range(n)])


def want_of(frames, params):
    status, streams, sizes = oracle.compress_frames(frames, oparams(params))
    assert (np.asarray(status) == 0).all()
    return streams


def same(out, nb, want):
    return all(nb[k] == len(w) and np.array_equal(out[k, :nb[k]], w) for k, w in enumerate(want))


@pytest.mark.parametrize("dense", [False, True])
@pytest.mark.parametrize("chunk", [1, 4])
@pytest.mark.parametrize("n", [1, 6])
def test_calls_after_stack_items_gave_up(dense, chunk, n):
    import torch
    frames = frames_of(n, seed=31)
    params = rb.default_params(atot_thr=300.0, lorenzo_dims=3, chunk_frames=chunk)
    want = want_of(frames, params)
    d = torch.from_numpy(frames).cuda()
    with rb.Context(GEOM, params, max_frames=n) as ctx:
        ctx.set_path(rb.PATH_FUSED)
        ctx.set_fused_dense_peaks(dense)
        for limit in LIMITS * 3:
            ctx.set_wait_limit(limit)
            out, nb, st = (t.cpu().numpy() for t in ctx.compress(d))
            assert np.isin(st, [rb.OK, rb.ERR_TIMEOUT]).all(), st
            assert (nb[st == rb.ERR_TIMEOUT] == 0).all()
            if limit == 0:
                assert (st == rb.ERR_TIMEOUT).all(), st
            if chunk == 1:  # else a frame's code is that of the frames of its chunk that did not give up
                for k in np.flatnonzero(st == rb.OK):
                    assert nb[k] == len(want[k]) and np.array_equal(out[k, :nb[k]], want[k]), (limit, k)
            ctx.set_wait_limit(-1)
            out, nb, st = (t.cpu().numpy() for t in ctx.compress(d))
            assert (st == rb.OK).all() and same(out, nb, want), limit


def test_joint_launch_after_stack_items_gave_up():
    import torch
    jobs = []
    for i, dims in enumerate((3, 2)):
        params = rb.default_params(atot_thr=300.0, lorenzo_dims=dims)
        f = frames_of(3, seed=40 + i)
        ctx = rb.Context(GEOM, params, max_frames=3)
        jobs.append(dict(ctx=ctx, frames=torch.from_numpy(f).cuda(), want=want_of(f, params),
                         out=torch.zeros((3, ctx.bound), dtype=torch.uint8, device="cuda"),
                         frame_bytes=torch.zeros(3, dtype=torch.int64, device="cuda"),
                         status=torch.zeros(3, dtype=torch.int32, device="cuda")))
    for limit in (0, 2, 20, -1):
        jobs[0]["ctx"].set_wait_limit(limit)
        with rb.Graph([{k: v for k, v in j.items() if k != "want"} for j in jobs], fused=True) as g:
            g.launch()
            torch.cuda.synchronize()
            st = jobs[0]["status"].cpu().numpy()
            assert np.isin(st, [rb.OK, rb.ERR_TIMEOUT]).all() and (limit != 0 or (st == rb.ERR_TIMEOUT).all())
            for j in jobs[1 if limit >= 0 else 0:]:
                assert (j["status"].cpu().numpy() == rb.OK).all()
                assert same(j["out"].cpu().numpy(), j["frame_bytes"].cpu().numpy(), j["want"]), limit
    for j in jobs:
        j["ctx"].close()
