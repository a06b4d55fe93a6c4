"""A launch that the CUDA runtime refuses is reported by the call that made it and
leaves no error behind for whoever asks the runtime next (the package and PyTorch
share one)."""
import ctypes

import numpy as np
import pytest

import paper_2206_11297_gb300 as rb
from synthetic import FrameRecipe, make_frame

pytestmark = pytest.mark.gpu


def runtime():
    for line in open("/proc/self/maps"):
        if "libcudart.so" in line:
            return ctypes.CDLL(line.split()[-1])
    pytest.skip("no shared CUDA runtime in this process")


@pytest.mark.parametrize("call", ["fused", "plain", "decompress", "static"])
def test_refused_launch_leaves_no_error(call):
    import torch
    geom, params = (2, 40, 44), rb.default_params(atot_thr=300.0)
    r = FrameRecipe(geom, peaks=("fixed", 4), seed=9)
    frames = torch.from_numpy(make_frame(r, 0)[None]).cuda()
    with rb.Context(geom, params, max_frames=1) as ctx:
        ctx.set_path(rb.PATH_FUSED if call == "fused" else rb.PATH_PLAIN)
        out, nb, st = ctx.compress(frames)
        offsets = torch.zeros(1, dtype=torch.int64, device="cuda")
        restored, rst = ctx.decompress(out.view(-1), offsets, 1)
        torch.cuda.synchronize()

        def run():
            if call == "decompress":
                ctx.decompress(out.view(-1), offsets, 1, out=restored, status=rst)
            elif call == "static":
                rb.compress_frame_static(geom, params, frames[0], out[0], nb, st)
            else:
                ctx.compress(frames, out=out, out_stride=out.shape[1], frame_bytes=nb, status=st)

        rt = runtime()
        captured, graph = ctypes.c_void_p(), ctypes.c_void_p()
        assert rt.cudaStreamCreate(ctypes.byref(captured)) == 0
        # while a stream that synchronises with the default one is captured, the
        # runtime refuses every launch on the default stream
        assert rt.cudaStreamBeginCapture(captured, 2) == 0
        try:
            with pytest.raises(rb.RoibinError) as e:
                run()
            left = rt.cudaPeekAtLastError()
        finally:
            rt.cudaStreamEndCapture(captured, ctypes.byref(graph))
            rt.cudaGetLastError()
            rt.cudaStreamDestroy(captured)
        assert e.value.code == rb.ERR_CUDA
        assert left == 0
        run()
        torch.cuda.synchronize()
        assert st.item() == rb.OK and rst.item() == rb.OK
        assert np.isfinite(restored.cpu().numpy()).all()
