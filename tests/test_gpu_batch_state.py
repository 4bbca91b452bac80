"""A batch's initial state (one kernel for all chains) and the read of a chain
into device memory, which waits once: the spins of hot and cold chains of the
smallest and of uneven sizes against the oracle, and a destination that is left
as it was once a device-side failure is recorded."""
import numpy as np
import pytest
import torch

import oracle
import paper_1105_5804_gb300 as sw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hot", [False, True])
def test_initial_state(hot):
    L, q = [4, 8, 100, 260, 12, 1028], [2, 127, 3, 2, 8, 5]
    seed = [3 + 2**33, 4, 5, 6, 7, 8]
    b = sw.sw_batch_create(L, q, [0.4] * 6, seed, sw.SW_CONV_AUTO, hot)
    try:
        for r in range(6):
            s = oracle.init_spins(L[r], q[r], seed[r], hot).reshape(-1)
            out = torch.full((L[r] * L[r] + 1,), -1, dtype=torch.int8, device="cuda")
            torch.cuda.synchronize()   # the batch copies on its own stream
            sw.sw_batch_get_spins(b, r, L[r], out[1:])   # a destination that is not 16-byte aligned
            assert np.array_equal(out[1:].cpu().numpy(), s) and int(out[0]) == -1, r
            assert np.array_equal(sw.sw_batch_get_spins(b, r, L[r]), s), r
            assert sw.sw_batch_observables(b, r, q[r]).shape[0] == 0
    finally:
        sw.sw_batch_destroy(b)


def test_failed_batch_leaves_the_destination():
    b = sw.sw_batch_create([64, 256], [2, 2], [0.4, 0.4], [1, 2], sw.SW_CONV_AUTO, True)
    try:
        out = torch.full((64 * 64,), 77, dtype=torch.int8, device="cuda")
        torch.cuda.synchronize()
        sw.sw_batch_set_schedule(b, sw.SW_BATCH_PERSISTENT)
        sw.sw_batch_set_barrier_limit(b, 0)
        sw.sw_batch_sweep(b, 1)
        for _ in range(2):
            with pytest.raises(sw.SwcclError) as e:
                sw.sw_batch_get_spins(b, 0, 64, out)
            assert e.value.code == sw.SW_ERR_TIMEOUT
        assert bool((out == 77).all())
    finally:
        sw.sw_batch_destroy(b)
