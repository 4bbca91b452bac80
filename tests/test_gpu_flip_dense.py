"""GPU parity of the flip where tiles have many roots (weak couplings down to
none: every site a root): more roots than the list holds, warps whose lanes
have unequal numbers of them, ragged tiles, every tile height, and batches."""
import numpy as np
import pytest

import oracle
import paper_1105_5804_gb300 as sw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [132, 260, 1024, 1284, 1300, 1536])
@pytest.mark.parametrize("q", [2, 3, 127])
@pytest.mark.parametrize("T", [0, 1 << 26, 1 << 29, 1 << 31])
def test_chain(L, q, T):
    h = sw.sw_create_threshold(L, q, T, 9, True)
    try:
        sw.sw_sweep(h, 2)
        s, obs = oracle.chain(L, q, T, 9, 0, 2, oracle.init_spins(L, q, 9, True))
        assert np.array_equal(sw.sw_get_spins(h), s)
        assert np.array_equal(sw.sw_observables(h, 4096), obs)
    finally:
        sw.sw_destroy(h)


@pytest.mark.parametrize("schedule", [sw.SW_BATCH_PHASES, sw.SW_BATCH_PERSISTENT])
@pytest.mark.parametrize("L", [[40, 260], [1300, 1024, 300]])
def test_batch(L, schedule):
    beta = [0.05 * (r + 1) for r in range(len(L))]
    b = sw.sw_batch_create(L, [2] * len(L), beta, list(range(len(L))), sw.SW_CONV_POTTS, True)
    try:
        sw.sw_batch_set_schedule(b, schedule)
        sw.sw_batch_sweep(b, 2)
        sw.sw_batch_sync(b)
        for r, x in enumerate(L):
            s, _ = oracle.chain(x, 2, oracle.threshold(beta[r]), r, 0, 2, oracle.init_spins(x, 2, r, True))
            assert np.array_equal(sw.sw_batch_get_spins(b, r, x), s), r
    finally:
        sw.sw_batch_destroy(b)
