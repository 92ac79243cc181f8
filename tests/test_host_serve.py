"""The served loop's host code against a CUDA runtime on host threads: calls
that may wait for the device never hold what a completion needs."""
import pytest

from tests.host_common import fake_library, run_against

SERVER = """
def server(slots=2, max_batch=4):
    d = L.ft_server_desc()
    L.ft_server_desc_default(C.byref(d))
    d.hbm_budget, d.n_slots, d.max_batch, d.slot_arena_bytes = 64 << 20, slots, max_batch, 8 << 20
    s = C.c_void_p()
    L.check(L.ft_server_create(C.byref(s), C.byref(d), None), 'server')
    return s

def open_stream(s, fr):
    sid = C.c_int(-1)
    L.check(L.ft_server_open_stream(s, C.byref(stream_desc_of(fr)), C.byref(sid)), 'open')
    return sid.value

def drain(s, n, limit=20.0):
    out, buf, t0 = [], (L.ft_completion * 64)(), time.time()
    while len(out) < n and time.time() - t0 < limit:
        k = L.ft_server_poll(s, buf, 64, 20000)
        out += [(buf[i].tag, buf[i].stream_id, buf[i].status) for i in range(k)]
    return out

frames = [scenes.pinhole_frame(i, W=320, H=240, n_left=200, n_map=300) for i in range(2)]
hosts = [HostFrame(f) for f in frames]
s = server()
a, b = open_stream(s, frames[0]), open_stream(s, frames[1])
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fake_library(tmp_path_factory)


# what a caller does while another stream's batch is running: each of these
# allocates, frees or copies in a way that waits for the device
CALLS = {
    "submit with images": "L.check(L.ft_server_submit(s, C.byref(hosts[1].request(b, 2, images=True)))); n = 2",
    "open": "open_stream(s, frames[1]); n = 1",
    "close": "L.check(L.ft_server_close_stream(s, b)); n = 1",
    "set map": "L.check(L.ft_server_set_map(s, b, C.byref(hosts[1].map_view()))); n = 1",
    "set pyramids": "p = hosts[1].pyramids(); L.check(L.ft_server_set_pyramids(s, b, C.byref(p[0]), C.byref(p[1]))); n = 1",
}


@pytest.mark.parametrize("call", list(CALLS))
def test_calls_that_wait_for_the_device_let_completions_through(fake, call):
    run_against(fake, SERVER + f"""
lib.fake_host_delay(100000)                 # a batch completes 0.1 s after its work
L.check(L.ft_server_submit(s, C.byref(hosts[0].request(a, 1))))
time.sleep(0.03)                            # the batch is on its stream
{CALLS[call]}
done = drain(s, n)
assert sorted(d[0] for d in done) == list(range(1, n + 1)), done
L.ft_server_destroy(s)
""", limit_s=30.0)


def test_streams_open_while_batches_launch(fake):
    # the table of streams grows (and moves) while the scheduler launches
    run_against(fake, SERVER + """
stop = []
def opener():
    d = stream_desc_of(scenes.pinhole_frame(3, W=64, H=48, n_left=4, n_map=4))
    while not stop:
        ids = []
        for _ in range(400):
            sid = C.c_int(-1)
            if L.ft_server_open_stream(s, C.byref(d), C.byref(sid)) == L.FT_OK: ids.append(sid.value)
        for i in ids: L.check(L.ft_server_close_stream(s, i))
t = threading.Thread(target=opener); t.start()
n = 0
while n < 300:
    for sid, h in ((a, hosts[0]), (b, hosts[1])):
        if L.ft_server_submit(s, C.byref(h.request(sid, n))) == L.FT_OK: n += 1
done = drain(s, n)
stop.append(1); t.join()
assert len(done) == n and all(d[2] == L.FT_OK for d in done)
L.ft_server_destroy(s)
""")


# the first memory copy of a launch, the kernels, the copy of the results (a
# launch of one request makes two copies), and the host function
@pytest.mark.parametrize("what,after", [("memcpy_async", 0), ("fused", 0), ("memcpy_async", 1), ("host_func", 0)])
def test_a_failed_launch_completes_its_requests(fake, what, after):
    run_against(fake, SERVER + f"""
lib.fake_fail({what!r}.encode(), {after})
L.check(L.ft_server_submit(s, C.byref(hosts[0].request(a, 1))))
assert drain(s, 1) == [(1, a, L.FT_ECUDA)]
st = L.ft_server_stats()
L.ft_server_get_stats(s, C.byref(st))
assert st.last_error == L.FT_ECUDA and st.completed == 1
for tag in range(2, 12):                    # the stream, its staging and both slots are free again
    for sid, h in ((a, hosts[0]), (b, hosts[1])):
        L.check(L.ft_server_submit(s, C.byref(h.request(sid, tag))))
    assert sorted(drain(s, 2)) == [(tag, a, L.FT_OK), (tag, b, L.FT_OK)]
L.check(L.ft_server_close_stream(s, a))
L.ft_server_destroy(s)
""")
