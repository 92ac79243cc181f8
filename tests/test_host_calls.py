"""The context's host code against a CUDA runtime on host threads: how a call's
table travels, which calls run as graphs, and that what a call that fails half way has enqueued keeps its
tables and its order."""
import pytest

from tests.host_common import fake_library, run_against

SETUP = """
def batch(n, seed, pyramids=False, fisheye=0, pose=False):
    fr = [scenes.pinhole_frame(seed + i, W=160, H=120, n_left=40, n_map=60) for i in range(n)]
    fr += [scenes.fisheye_frame(seed + i, n_left=150, n_map=60) for i in range(fisheye)]
    return PackedBatch(fr, device='cpu', pin=False, device_pyramids=pyramids, pose=pose)

ctx = Context(arena_bytes=64 << 20, max_frames=8)
a, b = stream(), stream()
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fake_library(tmp_path_factory)


def test_table_of_a_failed_call_stays_until_its_kernels_ran(fake):
    # the pyramid kernel of a call of two frames waits on its stream; the
    # fused kernel's launch fails; the fourth call after it takes the slot again
    run_against(fake, SETUP + """
two, three = batch(2, 1, pyramids=True), batch(3, 5)
gate = lib.fake_gate(a)
lib.fake_fail(b'fused', 0)
assert track(ctx, two, a) == L.FT_ECUDA
def more():
    for _ in range(4): L.check(track(ctx, three, a))
t = threading.Thread(target=more); t.start()
time.sleep(0.5)
lib.fake_open(gate)
t.join()
lib.cudaStreamSynchronize(a)
assert log() == ['pyramids 2'] + ['fused 3'] * 4, log()
ctx.close()
""")


@pytest.mark.parametrize("kind", ["several frames", "one frame"])
def test_calls_on_another_stream_come_after_a_failed_one(fake, kind):
    run_against(fake, SETUP + f"""
one = {kind == "one frame"}
first = batch(0, 1, fisheye=1) if one else batch(2, 1, pyramids=True)
gate = lib.fake_gate(a)
lib.fake_fail(b'fused', 0)
assert track(ctx, first, a) == L.FT_ECUDA
L.check(track(ctx, batch(3, 5), b))
time.sleep(0.3)
assert log() == [], log()
lib.fake_open(gate)
lib.cudaStreamSynchronize(a); lib.cudaStreamSynchronize(b)
assert log() == ['fisheye one' if one else 'pyramids 2', 'fused 3'], log()
ctx.close()
""")


@pytest.mark.parametrize("n,fisheye,pyramids,pose,kernels", [
    (2, 1, True, False, ["pyramids", "fisheye", "fused"]), (2, 1, True, True, ["pyramids", "fisheye", "fused", "pose"]),
    (3, 0, True, True, ["pyramids", "fused", "pose"]), (2, 1, False, True, ["fisheye", "fused", "pose"]),
    (2, 1, False, False, ["fisheye", "fused"]), (3, 0, False, False, ["fused"])])
def test_calls_of_three_kernels_run_as_graphs(fake, n, fisheye, pyramids, pose, kernels):
    # a graph per table slot and bucket, made at the slot's first call of the
    # kind and replayed for the other batches of the bucket
    run_against(fake, SETUP + f"""
g = Context(arena_bytes=64 << 20, max_frames=8, use_graphs=True)
first = batch({n}, 1, {pyramids}, {fisheye}, {pose})
other = batch({n} + 1, 7, {pyramids}, {fisheye}, {pose})
for _ in range(4): L.check(track(g, first, a))
for _ in range(4): L.check(track(g, other, a))
lib.cudaStreamSynchronize(a)
got = log()
graphs = {len(kernels)} > 2
assert got.count('graph made') == (4 if graphs else 0), got
assert got.count('graph') == (8 if graphs else 0), got
work = [x for x in got if not x.startswith('graph')]
assert work == [k + {f"' {n + fisheye}'"} for k in {kernels}] * 4 + [k + {f"' {n + 1 + fisheye}'"} for k in {kernels}] * 4, got
g.close()
""")


def test_table_of_a_lone_call_is_one_copy_on_its_stream(fake):
    # a stream with work takes the table from the context's own stream
    run_against(fake, SETUP + """
pb = batch(2, 1)
for _ in range(5):
    L.check(track(ctx, pb, a))
    lib.cudaStreamSynchronize(a)
assert lib.fake_table_kernels() == 0
gate = lib.fake_gate(a)
L.check(track(ctx, pb, a))
assert lib.fake_table_kernels() == 1
lib.fake_open(gate)
lib.cudaStreamSynchronize(a)
assert log() == ['fused 2'] * 6
ctx.close()
""")


@pytest.mark.parametrize("pyramids,fisheye,pose,kernels", [
    (False, 0, False, ["fused"]), (True, 0, False, ["pyramids", "fused"]), (True, 0, True, ["pyramids", "fused", "pose"]),
    (False, 1, False, ["fisheye", "fused"])])
def test_one_frame_travels_as_kernel_parameters(fake, pyramids, fisheye, pose, kernels):
    run_against(fake, SETUP + f"""
pb = batch({1 - fisheye}, 1, {pyramids}, {fisheye}, {pose})
gate = lib.fake_gate(a)
L.check(track(ctx, pb, a))
assert lib.fake_table_kernels() == 0
lib.fake_open(gate)
lib.cudaStreamSynchronize(a)
assert log() == [k + ' one' for k in {kernels}], log()
ctx.close()
""")


@pytest.mark.parametrize("ms,kept", [(0.9, "untuned"), (0.99, "listed"), (1.0, "listed"), (1.5, "listed")])
def test_autotuner_meets_the_untuned_shape(fake, ms, kept):
    # the launches' times by their strips: the shape an untuned call takes is
    # kept where it is clearly the fastest
    run_against(fake, SETUP + f"""
pb = batch(1, 1)
b = pb.batch()
def tuning():
    t = L.ft_tuning()
    L.check(L.ft_get_tuning(ctx.ptr, C.byref(b), C.byref(t)))
    return t
free = tuning()
assert free.strip_rows not in (16, 32, 64)
lib.fake_fast_strip.argtypes = [C.c_int, C.c_double]
lib.fake_fast_strip(free.strip_rows, {ms})
best = L.ft_tuning()
L.check(L.ft_autotune(ctx.ptr, a, None, C.byref(b), 2, C.byref(best)))
for t in (best, tuning()):
    if {kept == "untuned"}:
        assert (t.strip_rows, t.search_tile) == (free.strip_rows, free.search_tile), t.strip_rows
    else:
        assert t.strip_rows in (16, 32, 64), t.strip_rows
    assert t.ctas_per_sm in (1, 2, 3) and t.split_search in (1, -1)
""")


@pytest.mark.parametrize("W,H,right", [(752, 480, 1250), (640, 481, 600), (1280, 720, 4000), (320, 4000, 500), (64, 30, 9)])
def test_allocation_free_stereo_cuts_the_contexts_strips(fake, W, H, right):
    run_against(fake, SETUP + f"""
from paper_2509_10757_gb300.batch import pinhole_struct
pb = batch(1, 1)
fr, st, out = pb.frames[0], pb.stereo_frame(0), pb.stereo_out(0)
cam = pinhole_struct(fr.cam)
cam.width, cam.height, st.right.n = {W}, {H}, {right}
L.check(L.ft_stereo_match_pinhole(ctx.ptr, a, None, C.byref(cam), C.byref(st), C.byref(out)))
lib.cudaStreamSynchronize(a)
want = lib.fake_last_strip()
assert 0 < want <= 32
L.check(L.ft_stereo_match_pinhole_noalloc(a, None, C.byref(cam), C.byref(st), C.byref(out), None))
lib.cudaStreamSynchronize(a)
assert log() == ['fused one', 'fused 1'] and lib.fake_last_strip() == want
ctx.close()
""")
