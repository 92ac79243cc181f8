"""Forms of a call that the other GPU tests do not reach: the largest batch."""
import ctypes as C

import numpy as np
import pytest

import oracle as orc
from paper_2509_10757_gb300 import scenes
from tests.gpu_common import assert_fisheye_equal, assert_search_equal

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

P = dict(scenes.DEFAULT_PARAMS)


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2509_10757_gb300 import build
    build.build()
    from paper_2509_10757_gb300 import _lib as L
    return L


def test_largest_batch_of_fisheye_frames(lib):
    # 65536 frames, as many as a context takes: the frame of the first half
    # and the frame of the second share their buffers, so every frame's outputs
    # are the oracle's
    from paper_2509_10757_gb300.batch import Context, PackedBatch, stream_handle
    frames = [scenes.fisheye_frame(s, n_left=24, n_map=20) for s in (51, 52)]
    pb = PackedBatch(frames)
    pb.upload()
    pb.clear_outputs()
    n = 65536
    jobs = (lib.ft_frame_job * n)(*([pb.jobs[0]] * (n // 2) + [pb.jobs[1]] * (n // 2)))
    b = lib.ft_batch()
    b.n, b.frames = n, C.cast(jobs, C.POINTER(lib.ft_frame_job))
    c = Context(arena_bytes=4 << 30, max_frames=n)
    try:
        lib.check(lib.ft_track_batch(c.ptr, stream_handle(), None, C.byref(b)), "ft_track_batch")
        pb.download()
        assert c.sync_status() == 0
    finally:
        c.close()
    for f, fr in enumerate(frames):
        st, se = orc.track_frame(P, fr)
        assert (st["r_idx"] >= 0).sum() > 3
        out = pb.outputs(f)
        assert_fisheye_equal(out, st, f"frame {f}: ")
        assert_search_equal(out, se, "l", "l", f"frame {f}: ")
        assert_search_equal(out, se, "r", "r", f"frame {f}: ")
