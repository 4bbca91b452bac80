"""Host code of the library on a fake CUDA runtime (fake_cudart.cpp): what the
C entries enqueue, refuse and count, without a GPU."""
import ctypes

import numpy as np
import pytest

import host_runtime

SW_OK, SW_ERR_CUDA = 0, 3


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return host_runtime.load(tmp_path_factory.mktemp("fake"))


def _ptr(n):
    """A device buffer of the fake runtime (kernels do not run)."""
    a = np.zeros(n, np.uint8)
    return a, a.ctypes.data_as(ctypes.c_void_p)


def _batch(fake, L, stream, q=3):
    n = len(L)
    q, beta, seed = np.full(n, q, np.int32), np.full(n, 0.7), np.arange(n, dtype=np.uint64)
    L = np.asarray(L, np.int32)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    need = fake.sw_batch_device_bytes(n, p(L), p(q))
    raw = np.zeros(need + 256, np.uint8)
    ws = raw[-raw.ctypes.data % 256:][:need]
    b = fake.sw_batch_create_ws(n, p(L), p(q), p(beta), p(seed), 0, 1, p(ws), need, stream)
    assert b, fake.sw_last_error()
    return b, ws


@pytest.mark.parametrize("L", [[16], [64, 100, 300], [512] * 40])
def test_batch_tables_outlive_their_copy(fake, L):
    """sw_batch_create_ws returns without waiting: what it copies to the device
    is the batch's to keep until the copy is made."""
    st = fake.fake_stream(0)
    b, ws = _batch(fake, L, st)
    assert fake.cudaStreamSynchronize(st) == 0
    sweep, obs_done = ws[:16].view(np.int64)        # the control block
    assert (sweep, obs_done) == (0, -1)
    tiles = [-(-x // 32) * -(-x // 256) for x in L]
    info = (ctypes.c_int64 * 8)()
    fake.sw_batch_info(b, info)
    assert info[2] == sum(tiles)
    tile_map = np.repeat(np.arange(len(L), dtype=np.int32), tiles)
    starts = range(512, len(ws) - tile_map.nbytes, 256)   # after the control block and the chain table
    at = next(k for k in starts if np.array_equal(ws[k:k + tile_map.nbytes].view(np.int32), tile_map))
    first_chain = at + -(-tile_map.nbytes // 256) * 256
    assert ws[256:264].view(np.uint64)[0] == ws.ctypes.data + first_chain   # chain 0: its spins
    fake.sw_batch_destroy(b)


@pytest.mark.parametrize("failing", [1, 2, 3])
def test_a_failed_launch_leaves_no_pending_error(fake, failing):
    """A failed launch is the call's to report; the caller's next
    cudaGetLastError does not find it again."""
    st = fake.fake_stream(0)
    mask, m = _ptr(1024)
    lab, l = _ptr(4 * 4096)
    h = fake.sw_create_threshold(256, 2, 1 << 31, 1, 1, st)
    h3 = fake.sw3_create(40, 9, 20, 2, 1 << 31, 1, 1, st)
    for call in (lambda: fake.ccl_label(m, l, 64, 64, 1, st), lambda: fake.sw_sweep(h, 1), lambda: fake.sw3_sweep(h3, 1)):
        fake.fake_fail_launch(failing)
        assert call() == SW_ERR_CUDA and fake.sw_last_error()
        assert fake.cudaGetLastError() == 0
    fake.sw_destroy(h)
    fake.sw3_destroy(h3)


@pytest.mark.parametrize("L,tiles", [([16], 1), ([16, 100, 300], 24), ([2048] * 3, 1536)])
def test_a_batch_is_set_up_by_many_blocks(fake, L, tiles):
    """Its observable rings (4 MB a chain for q = 127) take more than a block
    per tile if the tiles are few."""
    st = fake.fake_stream(0)
    b, ws = _batch(fake, L, st, q=127)
    c = (ctypes.c_longlong * 5)()
    fake.fake_counts(c)
    assert c[3] == tiles * max(1, min(64, 1216 // tiles))
    fake.sw_batch_destroy(b)


def _counts(fake):
    c = (ctypes.c_longlong * 5)()
    fake.fake_counts(c)
    return list(c)[:3]


def _sweeps(info, h, k):
    v = (ctypes.c_int64 * 8)()
    info(h, v)
    return v[k]


@pytest.mark.parametrize("L", [64, 256, 2048])
@pytest.mark.parametrize("mode", ["fused", "staged", "few"])
@pytest.mark.parametrize("timing", [0, 1])
@pytest.mark.parametrize("call", ["sweep", "io"])
def test_captured_sweeps_are_refused_before_anything_is_enqueued(fake, L, mode, timing, call):
    st = fake.fake_stream(0)
    h = fake.sw_create_threshold(L, 2, 1 << 31, 1, 1, st)
    if mode == "staged":
        fake.sw_set_mode(h, 0)
    elif mode == "few":
        fake.sw_set_update(h, 1, 4, 1 << 31)
    fake.sw_set_timing(h, timing)
    _, spins = _ptr(L * L)
    run = (lambda: fake.sw_sweep(h, 3)) if call == "sweep" else (lambda: fake.sw_sweep_io(h, spins, 3, None, spins))
    for warm in range(2):
        before = _counts(fake)
        fake.fake_capture(st, 1)
        assert run() == SW_ERR_CUDA and b"captured" in fake.sw_last_error()
        assert _counts(fake) == before and fake.fake_capture_valid(st)
        fake.fake_capture(st, 0)
        assert fake.cudaGetLastError() == 0
        assert _sweeps(fake.sw_get_info, h, 4) == 3 * warm
        assert run() == SW_OK
    if mode == "fused" and L > 112:   # the sweeps' last observables are still to be counted when they are read
        before = _counts(fake)[0]
        fake.fake_capture(st, 1)
        run()
        fake.fake_capture(st, 0)
        n, rows = ctypes.c_int(), (ctypes.c_int64 * 18)()
        assert fake.sw_observables(h, rows, 6, ctypes.byref(n)) == SW_OK and n.value == 6
        assert _counts(fake)[0] > before + 2   # counted, then read: status and rows
    fake.sw_destroy(h)


@pytest.mark.parametrize("timing", [0, 1])
def test_captured_cubic_sweeps_are_refused(fake, timing):
    st = fake.fake_stream(0)
    h = fake.sw3_create(40, 9, 20, 2, 1 << 31, 1, 1, st)
    fake.sw3_set_timing(h, timing)
    for warm in range(2):
        before = _counts(fake)
        fake.fake_capture(st, 1)
        assert fake.sw3_sweep(h, 2) == SW_ERR_CUDA
        assert _counts(fake) == before and fake.fake_capture_valid(st)
        fake.fake_capture(st, 0)
        assert _sweeps(fake.sw3_get_info, h, 6) == 2 * warm
        assert fake.sw3_sweep(h, 2) == SW_OK
    fake.sw3_destroy(h)


@pytest.mark.parametrize("graph", [0, 1])
def test_batch_sweeps_in_a_capture(fake, graph):
    """They go into it as direct launches and leave the batch's own graph for
    later; a batch that replays its graph already refuses, and the capture goes
    on."""
    st = fake.fake_stream(0)
    b, ws = _batch(fake, [64, 300], st)
    fake.sw_batch_set_graph(b, graph)
    fake.fake_capture(st, 1)
    before = _counts(fake)
    assert fake.sw_batch_sweep(b, 2) == SW_OK
    after = _counts(fake)
    assert after[1] - before[1] == 6 and after[2] == before[2] and fake.fake_capture_valid(st)
    fake.fake_capture(st, 0)
    assert fake.sw_batch_sweep(b, 2) == SW_OK
    assert _counts(fake)[2] - after[2] == 2 * graph and _sweeps(fake.sw_batch_info, b, 6) == graph
    fake.fake_capture(st, 1)
    assert fake.sw_batch_sweep(b, 1) == (SW_ERR_CUDA if graph else SW_OK)
    assert fake.fake_capture_valid(st) and _sweeps(fake.sw_batch_info, b, 3) == (4 if graph else 5)
    fake.fake_capture(st, 0)
    fake.sw_batch_destroy(b)


@pytest.mark.parametrize("L", [64, 256, 2048])
@pytest.mark.parametrize("timing", [0, 1])
def test_sweeps_enqueued_while_another_device_is_current(fake, L, timing):
    st = fake.fake_stream(1)
    fake.fake_set_device(1)
    h = fake.sw_create_threshold(L, 2, 1 << 31, 1, 1, st)
    h3 = fake.sw3_create(40, 9, 20, 2, 1 << 31, 1, 1, st)
    fake.sw_set_timing(h, timing)
    fake.sw3_set_timing(h3, timing)
    for warm in range(2):
        fake.fake_set_device(0)
        assert fake.sw_sweep(h, 3) == SW_OK, fake.sw_last_error()
        assert fake.sw3_sweep(h3, 3) == SW_OK, fake.sw_last_error()
        assert fake.fake_device() == 0 and fake.cudaGetLastError() == 0
    assert _sweeps(fake.sw_get_info, h, 4) == _sweeps(fake.sw3_get_info, h3, 6) == 6
    fake.sw_destroy(h)
    fake.sw3_destroy(h3)


def test_noalloc_loads_every_kernel_on_its_first_call(tmp_path):
    """The first call on a device may take device memory and time; later ones,
    of any size, launch only what is loaded."""
    fake = host_runtime.load(tmp_path)   # a library of its own: nothing loaded yet
    st = fake.fake_stream(0)
    mask, m = _ptr(1 << 20)
    lab, l = _ptr(1 << 24)
    cold = lambda: (lambda c: (fake.fake_counts(c), c[4])[1])((ctypes.c_longlong * 5)())
    assert fake.ccl_label_noalloc(m, l, 1, 1, 1, st) == SW_OK, fake.sw_last_error()
    assert cold() == 0
    for H, W in [(200, 300), (1000, 1200), (1500, 1500), (2000, 2000)]:
        assert fake.ccl_label_noalloc(m, l, H, W, 0, st) == SW_OK, fake.sw_last_error()
    assert cold() == 0


@pytest.mark.parametrize("q,line", [(2, 112), (3, 112), (4, 96), (8, 96), (9, 96), (127, 96)])
def test_where_the_one_block_kernel_ends(fake, q, line):
    """Up to the line all sweeps of a call are one launch, past it three each."""
    st = fake.fake_stream(0)
    for L, launches in ((4, 1), (line, 1), (line + 4, 30)):
        h = fake.sw_create_threshold(L, q, 1 << 31, 1, 1, st)
        before = _counts(fake)[0]
        assert fake.sw_sweep(h, 10) == SW_OK
        assert _counts(fake)[0] - before == launches, L
        fake.sw_destroy(h)
