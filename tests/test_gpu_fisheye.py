"""Fisheye matching where blocks of a cluster have no columns: the blocks
other than the first go from their rows straight to the exchange of the row
minima, in the calls that split a row's columns over two or four blocks.
Compared with the CPU oracle bit for bit."""
import numpy as np
import pytest

import oracle as orc
from paper_2509_10757_gb300 import scenes
from tests.gpu_common import assert_fisheye_equal
from tests.test_gpu_parity import _shrink, run_fused

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

P = dict(scenes.DEFAULT_PARAMS)


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2509_10757_gb300 import build
    build.build()
    from paper_2509_10757_gb300.batch import Context
    c = Context(arena_bytes=256 << 20, max_frames=16)
    yield c
    c.close()


# right keypoints in the overlap: none of them all, none in it, one step of 128
# columns (three blocks without), two, three and four and a remainder
@pytest.mark.parametrize("inside", [None, 0, 1, 128, 129, 384, 513])
@pytest.mark.parametrize("nl", [1, 129, 2500])
def test_blocks_without_columns(ctx, inside, nl):
    from paper_2509_10757_gb300.batch import PackedBatch, run_stereo
    fr = _shrink(scenes.fisheye_frame(81, n_left=2500, n_map=0), nl=nl, nr=0 if inside is None else None)
    rig = fr.rig
    out_x = np.float32(rig.lap_r1 + 50.0)
    if inside is not None:
        fr.right.x[:] = out_x
        fr.right.x[200:200 + inside] = np.linspace(rig.lap_r0, rig.lap_r1, inside, dtype=np.float32)
    ref = orc.stereo_frame(P, fr)
    n_in = int(np.count_nonzero((fr.right.x >= rig.lap_r0) & (fr.right.x <= rig.lap_r1)))
    assert n_in == (inside or 0)
    pb = PackedBatch([fr])
    pb.upload()
    for _ in range(3):
        pb.clear_outputs()
        run_stereo(ctx, pb, 0)
    pb.download()
    assert ctx.sync_status() == 0
    assert_fisheye_equal(pb.outputs(0), ref, f"{nl} left, {inside} in the overlap, alone: ")
    for n in (2, 5):
        many = run_fused(ctx, [fr] * n)
        for f in range(n):
            assert_fisheye_equal(many.outputs(f), ref, f"{nl} left, {inside} in the overlap, frame {f} of {n}: ")


@pytest.mark.parametrize("n", [1, 3])
def test_waits_that_run_out_leave_a_usable_context(ctx, n):
    # a bound of 1 ns on the waits for products: whether or not one runs out,
    # the call ends, its outputs are defined (a right keypoint or none) and the
    # next call's results are the oracle's
    from paper_2509_10757_gb300 import _lib as L
    from paper_2509_10757_gb300.batch import PackedBatch, run_batch
    fr = scenes.fisheye_frame(82, n_left=2500, n_map=0)
    ref = orc.stereo_frame(P, fr)
    pb = PackedBatch([fr] * n)
    pb.upload()
    try:
        for _ in range(20):
            L.check(L.ft_set_debug(ctx.ptr, 0, 1), "debug")
            pb.clear_outputs()
            run_batch(ctx, pb)
            status = ctx.sync_status()
            assert status in (L.FT_OK, L.FT_ETIMEOUT)
            pb.download()
            for f in range(n):
                out = pb.outputs(f)
                assert out["r_idx"].min() >= -1 and out["r_idx"].max() < fr.right.n
                assert out["d1"].min() >= -1 and out["d2"].max() <= 256
    finally:
        L.check(L.ft_set_debug(ctx.ptr, 0, 0), "debug")
    pb.clear_outputs()
    run_batch(ctx, pb)
    pb.download()
    assert ctx.sync_status() == L.FT_OK
    for f in range(n):
        assert_fisheye_equal(pb.outputs(f), ref, f"after the short waits, frame {f} of {n}: ")
