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


def _batch(fake, L, stream):
    n = len(L)
    q, beta, seed = np.full(n, 3, np.int32), np.full(n, 0.7), np.arange(n, dtype=np.uint64)
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
