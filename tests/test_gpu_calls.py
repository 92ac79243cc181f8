"""Forms of a call that the other GPU tests do not reach: the largest batch, and
graphs with a node of every kernel replayed for other batches of their bucket.
Compared with the CPU oracle."""
import copy
import ctypes as C

import numpy as np
import pytest

import oracle as orc
from paper_2509_10757_gb300 import scenes
from tests.gpu_common import assert_fisheye_equal, assert_search_equal, assert_stereo_equal
from tests.test_gpu_parity import _shrink, _with_oracle_pyramids, check_frame
from tests.test_gpu_pose import check_pose

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


@pytest.mark.parametrize("pose", [False, True])
def test_graphs_replay_other_batches_of_their_bucket(lib, pose):
    # three kernels or four with a fisheye node among them (such calls run as
    # graphs: test_host_calls): three frames, then four with other counts of
    # keypoints and points, in turn through all table slots twice and again
    from paper_2509_10757_gb300.batch import Context, PackedBatch, run_batch
    q = scenes.fisheye_frame(61, n_left=1500, n_map=4000)
    groups = [[scenes.single_pinhole(61), q, scenes.single_pinhole(62)],
              [_shrink(q, nl=1100, nr=700, m=2100), _shrink(scenes.single_pinhole(63), nl=1100, m=2500),
               scenes.single_pinhole(64), _shrink(scenes.fisheye_frame(62, n_left=1500, n_map=3000), nr=0)]]
    pbs = [PackedBatch(g, device_pyramids=True, pose=pose) for g in groups]
    c = Context(arena_bytes=256 << 20, max_frames=8, use_graphs=True)
    runs = []
    try:
        for pb in pbs:
            pb.upload()
        for i in range(18):
            pb = pbs[i % 2]
            pb.clear_outputs()
            run_batch(c, pb)
            if i >= 14:
                pb.download()
                runs.append(pb.host_out.numpy().copy())
        assert c.sync_status() == 0
    finally:
        c.close()
    for k in (0, 1):
        assert np.array_equal(runs[k], runs[k + 2])
        for f, fr in enumerate(groups[k]):
            out = pbs[k].outputs(f)
            if fr.camera == "fisheye":
                check_frame(pbs[k], f, what=f"graph of group {k}")
                continue
            fr = _with_oracle_pyramids(fr)
            st, se = orc.track_frame(P, fr)
            assert_search_equal(out, se, "l", None, f"graph of group {k}, frame {f}: ")
            if pose:
                ref = orc.optimize_pose(P, fr.cam, fr.pose, fr.left, st["u_right"], fr.map.pos, se["mp_kp"])
                check_pose(out, ref, f"graph of group {k}, frame {f}: ")


@pytest.mark.parametrize("kind,mode", [("pinhole", "global"), ("fisheye", "global"), ("two", "relaxed"),
                                       ("pyramids and pose", "relaxed")])
def test_calls_captured_into_a_callers_graph(lib, kind, mode):
    # a captured call replays with the inputs its buffers hold then: a frame's
    # own, another's, its own again, with other calls of the context between
    from paper_2509_10757_gb300.batch import Context, PackedBatch, run_batch
    # (the pose and the cameras are part of the call: the other frame has the same)
    fr = scenes.fisheye_frame(65) if kind == "fisheye" else scenes.single_pinhole(65)
    other = copy.deepcopy(fr)
    other.right.desc[::3] ^= 0xff
    other.map.desc[::3] ^= 0xff
    more = [scenes.fisheye_frame(67)] if kind == "two" else [scenes.single_pinhole(67)] if "pose" in kind else []
    kw = dict(device_pyramids=True, pose=True) if "pose" in kind else {}
    a, b = PackedBatch([fr] + more, **kw), PackedBatch([other] + more, **kw)
    assert a.lin.size == b.lin.size and a.lout.size == b.lout.size
    c = Context(arena_bytes=256 << 20, max_frames=8)
    try:
        # (all the context's calls on one stream: a captured call cannot wait
        # for one outside the capture)
        s = torch.cuda.Stream()
        want = []
        for pb in (a, b):
            pb.upload()
            pb.clear_outputs()
            torch.cuda.synchronize()
            run_batch(c, pb, stream=s)
            pb.download()
            want.append(pb.host_out.numpy().copy())
        if not kw:
            check_frame(a, 0, what="before the capture")
        assert not np.array_equal(*want)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s, capture_error_mode=mode):
            run_batch(c, a, stream=s)
        for k, src in ((0, a), (1, b), (0, a)):
            a.dev_in.copy_(src.host_in)
            a.clear_outputs()
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            a.download()
            assert np.array_equal(a.host_out.numpy(), want[k])
            run_batch(c, b, stream=s)
        torch.cuda.synchronize()
        assert c.sync_status() == 0
    finally:
        c.close()


@pytest.mark.parametrize("W,H", [(752, 480), (401, 301), (64, 48)])
def test_one_frame_with_its_pyramids_built(lib, W, H):
    # one frame travels as kernel parameters, its pyramids' kernel included:
    # levels, matches and pose, other calls of the context in between
    from paper_2509_10757_gb300.batch import Context, PackedBatch, run_batch
    fr = scenes.pinhole_frame(68, W=W, H=H, n_left=min(600, W * H // 60), n_map=800)
    other = PackedBatch([scenes.single_pinhole(69), scenes.fisheye_frame(69)])
    other.upload()
    pb = PackedBatch([fr], device_pyramids=True, pose=True)
    pb.upload()
    c = Context(arena_bytes=256 << 20, max_frames=4)
    try:
        for _ in range(3):
            pb.dev_pyr.fill_(0x5a)
            pb.clear_outputs()
            n = c.launches()
            run_batch(c, pb)
            assert c.launches() - n == 3
            run_batch(c, other)
        pb.download()
        assert c.sync_status() == 0
    finally:
        c.close()
    fr = _with_oracle_pyramids(fr)
    for side, levels in (("L", fr.pyr_left), ("R", fr.pyr_right)):
        for l in range(1, len(levels)):
            assert np.array_equal(pb.device_level(0, side, l), levels[l]), (side, l)
    st, se = orc.track_frame(P, fr)
    out = pb.outputs(0)
    assert_stereo_equal(out, st)
    assert_search_equal(out, se, "l")
    ref = orc.optimize_pose(P, fr.cam, fr.pose, fr.left, st["u_right"], fr.map.pos, se["mp_kp"])
    check_pose(out, ref, f"{W}x{H}: ")


@pytest.mark.parametrize("strip", [4, 24, 48])
@pytest.mark.parametrize("tile", [256, 1024])
@pytest.mark.parametrize("split", [1, -1])
def test_shapes_of_untuned_calls(lib, strip, tile, split):
    # the strip heights, search tiles and search forms the launch rule picks,
    # on frames it does not pick them for
    from paper_2509_10757_gb300.batch import Context, PackedBatch, run_batch
    pb = PackedBatch([scenes.single_pinhole(70), scenes.fisheye_frame(70),
                      scenes.pinhole_frame(70, W=1280, H=720, n_left=3000, n_map=5000)])
    pb.upload()
    pb.clear_outputs()
    c = Context(arena_bytes=256 << 20, max_frames=4)
    try:
        b = pb.batch()
        t = lib.ft_tuning(strip_rows=strip, search_tile=tile, resolve_tile=2048, split_search=split)
        lib.check(lib.ft_set_tuning(c.ptr, C.byref(b), C.byref(t)), "ft_set_tuning")
        run_batch(c, pb)
        pb.download()
        assert c.sync_status() == 0
    finally:
        c.close()
    for f in range(3):
        check_frame(pb, f, what=f"strips of {strip}, tiles of {tile}, split {split}")
