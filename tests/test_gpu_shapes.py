"""GPU parity at the sizes where the kernels change form: tile and chunk
edges, remainders, the smallest and largest case of each branch, and the call
forms (one frame, batch, graph, several streams, a small arena) against each
other.  Every comparison is with the CPU oracle: whole numbers, projections
and triangulations bit for bit (gpu_common), poses within the bound that
test_gpu_pose derives."""
import ctypes as C

import numpy as np
import pytest

import oracle as orc
from paper_2509_10757_gb300 import scenes
from tests.gpu_common import assert_fisheye_equal, assert_search_equal
from tests.test_gpu_orb import assert_orb_equal, extract
from tests.test_gpu_parity import _shrink, _with_oracle_pyramids, check_frame, run_fused
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


@pytest.fixture(scope="module")
def ctx(lib):
    from paper_2509_10757_gb300.batch import Context
    c = Context(arena_bytes=1 << 30, max_frames=64)
    yield c
    c.close()


@pytest.mark.parametrize("n", [8527, 8528, 8529, 17057, 65537])
def test_search_over_grids_in_several_parts(ctx, lib, n):
    # the search keeps 8528 of a camera's packed grid entries on chip at a
    # time; above 65535 keypoints the entries hold 32-bit indices
    from paper_2509_10757_gb300.batch import PackedBatch, run_search
    fr = scenes.pinhole_frame(72, 1280, 720, n, 0.0, 0.05, 1500)
    pb = PackedBatch([fr])
    pb.upload()
    pb.clear_outputs()
    run_search(ctx, pb, 0, u_right=False)
    pb.download()
    assert ctx.sync_status() == 0
    ref = orc.search_frame(P, fr, None)
    assert (ref["mp_kp"] >= 0).sum() > 100
    assert_search_equal(pb.outputs(0), ref, "l", None, f"{n} keypoints: ")


POSE_COUNTS = [0, 1, 2, 127, 128, 129, 511, 512, 513, 8191, 8192, 8193]


def test_pose_over_numbers_of_observations(ctx, lib):
    # 512 threads a frame over four blocks, 8192 observations on chip, the
    # list in device memory beyond
    from paper_2509_10757_gb300.batch import PackedBatch, run_pose
    fr = scenes.pinhole_frame(71, 752, 480, 9000, 0.1, 0.05, 15100)
    pick = fr.truth["map_kp"]
    pb = PackedBatch([fr], pose=True)
    pb.upload()
    at = pb.pout(0, "mp_kp_l") - pb.out_base
    for n in POSE_COUNTS:
        mk = np.full(fr.map.n, -1, np.int32)
        mk[:n] = pick[:n]
        pb.clear_outputs()
        pb.dev_out[at:at + mk.nbytes].copy_(torch.from_numpy(mk.view(np.uint8)))
        run_pose(ctx, pb, 0, u_right=False)
        pb.download()
        assert ctx.sync_status() == 0
        ref = orc.optimize_pose(P, fr.cam, fr.pose, fr.left, None, fr.map.pos, mk)
        check_pose(pb.outputs(0), ref, f"{n} observations: ")


FISHEYE_SIZES = [(1, 1), (1, 300), (127, 129), (128, 128), (129, 127), (300, 1), (300, 2047), (300, 2048),
                 (300, 2049), (2047, 300), (2500, 2500)]


@pytest.mark.parametrize("equal", [False, True])
def test_fisheye_matching_at_tile_edges(ctx, lib, equal):
    # tiles of 128 left keypoints, a window of 2048 right ones, the right
    # keypoints split over 1, 2 or 4 blocks by the size of the call: each
    # frame alone (4 blocks for the smaller ones), all together, and several
    # times over (1 block); equal descriptors tie every distance
    from paper_2509_10757_gb300.batch import PackedBatch, run_stereo
    base = scenes.fisheye_frame(73, n_left=2600, n_map=0)
    if equal:
        base.left.desc[:] = base.left.desc[0]
        base.right.desc[:] = base.left.desc[0]
    frames = [_shrink(base, nl=nl, nr=nr) for nl, nr in FISHEYE_SIZES]
    refs = [orc.stereo_frame(P, fr) for fr in frames]
    pb = PackedBatch(frames)
    pb.upload()
    pb.clear_outputs()
    for f in range(len(frames)):
        run_stereo(ctx, pb, f)
    pb.download()
    assert ctx.sync_status() == 0
    many = run_fused(ctx, frames * 3)
    few = run_fused(ctx, frames)
    for f, size in enumerate(FISHEYE_SIZES):
        for out, what in ((pb, "alone"), (few, "batch"), (many, "large batch")):
            assert_fisheye_equal(out.outputs(f), refs[f], f"{size} {what}: ")


@pytest.mark.parametrize("shape", [(41, 300), (62, 60), (63, 61), (124, 90), (125, 91), (187, 44)])
def test_extraction_at_tile_edges(ctx, lib, shape):
    # tiles of 62 x 30 pixels: level 0 at and one past multiples of them, and
    # levels smaller than a tile or without a pixel inside the border
    rng = np.random.default_rng(shape[0])
    img = scenes.band_limited_noise(rng, shape[1], shape[0], sigma=1.2).astype(np.uint8)
    lv = scenes.build_pyramid(img)
    caps, pat = [60, 40, 30, 20, 10, 10, 5, 5], scenes.orb_pattern()
    ref = orc.extract_orb(P, lv, 10, 19, caps, pat)
    got = extract(ctx, lib, [lv, lv], caps, pat, 10, 19)
    for i in range(2):
        assert_orb_equal(got[i], ref, f"{shape} image {i}: ")


@pytest.mark.parametrize("cap", [300, 512, 513, 1500, 4095, 4096])
def test_extraction_selects_among_equal_scores(ctx, lib, cap):
    # 5040 corners of one score on level 0: the selection falls to the raster
    # order alone, below and above its 512 sorted in one step
    img = np.full((480, 752), 90, np.uint8)
    img[4::8, 4::8] = img[4::8, 5::8] = 200
    lv = scenes.build_pyramid(img)
    pat = scenes.orb_pattern()
    ref = orc.extract_orb(P, lv, 20, 19, [cap] * 8, pat)
    assert ref["n_level"][0] == cap
    assert_orb_equal(extract(ctx, lib, [lv], [cap] * 8, pat)[0], ref, f"cap {cap}: ")


def test_one_frame_calls_repeat_and_alternate(ctx, lib):
    # one-frame calls keep their queue and counters in a few words that the
    # last block leaves zero: the same call again, other frames in between
    from paper_2509_10757_gb300.batch import PackedBatch, run_batch
    frames = [scenes.single_pinhole(31), scenes.fisheye_frame(31), _shrink(scenes.single_pinhole(32), m=0)]
    pbs = [PackedBatch([fr]) for fr in frames]
    for pb in pbs:
        pb.upload()
    for _ in range(3):
        for pb in pbs:
            pb.clear_outputs()
            run_batch(ctx, pb)
        for pb in pbs:
            pb.download()
        assert ctx.sync_status() == 0
        for pb in pbs:
            check_frame(pb, 0, what="one frame, alternating")


@pytest.mark.parametrize("graphs", [False, True])
def test_calls_in_flight_on_two_streams(lib, graphs):
    # more calls than table slots, of different frames and kinds, on two
    # streams in turn without a synchronisation between them
    from paper_2509_10757_gb300.batch import Context, PackedBatch, run_batch
    groups = [[scenes.single_pinhole(33), scenes.fisheye_frame(33)], [scenes.fisheye_frame(34)],
              [scenes.single_pinhole(35), scenes.single_pinhole(36), scenes.single_pinhole(37)]]
    pbs = [PackedBatch(g, device_pyramids=i == 2, pose=i == 2) for i, g in enumerate(groups)]
    for pb in pbs:
        pb.upload()
        pb.clear_outputs()
    c = Context(arena_bytes=256 << 20, max_frames=8, use_graphs=graphs)
    try:
        streams = [torch.cuda.Stream(), torch.cuda.Stream()]
        torch.cuda.synchronize()
        for i in range(14):
            run_batch(c, pbs[i % 3], stream=streams[i % 2])
        torch.cuda.synchronize()
        assert c.sync_status() == 0
    finally:
        c.close()
    for pb in pbs[:2]:
        pb.download()
        for f in range(len(pb.frames)):
            check_frame(pb, f, what="two streams")
    # the third group's levels are the library's own resampling
    pbs[2].download()
    for f, fr in enumerate(pbs[2].frames):
        fr = _with_oracle_pyramids(fr)
        st, se = orc.track_frame(P, fr)
        assert_search_equal(pbs[2].outputs(f), se, "l", None, f"device pyramids frame {f}: ")
        ref = orc.optimize_pose(P, fr.cam, fr.pose, fr.left, st["u_right"], fr.map.pos, se["mp_kp"])
        check_pose(pbs[2].outputs(f), ref, f"device pyramids frame {f}: ")


def test_smallest_arena_gives_the_same_results(lib):
    # the launch rule takes the two-pass search for a small batch; its extra
    # scratch is given up where the arena has no room for it
    from paper_2509_10757_gb300.batch import Context, PackedBatch, stream_handle
    frames = scenes.pinhole_batch(seed=38, n_frames=16)
    pb = PackedBatch(frames)
    pb.upload()
    b = pb.batch()

    def status(arena):
        c = Context(arena_bytes=arena, max_frames=16)
        try:
            r = c.lib.ft_track_batch(c.ptr, stream_handle(), None, C.byref(b))
            torch.cuda.synchronize()
            assert r != 0 or c.sync_status() == 0
            return r
        finally:
            c.close()

    lo, hi = 1 << 16, 64 << 20
    assert status(hi) == 0
    while hi - lo > 4096:
        mid = (lo + hi) // 2
        r = status(mid)
        assert r in (lib.FT_OK, lib.FT_ENOMEM)
        lo, hi = (lo, mid) if r == 0 else (mid, hi)
    assert status(lo) == lib.FT_ENOMEM
    pb.clear_outputs()
    assert status(hi) == 0
    pb.download()
    for f in range(len(frames)):
        check_frame(pb, f, what="smallest arena")
