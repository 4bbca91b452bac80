"""GPU parity of batches on tiles of 8 and 16 rows (batches with few tiles)
against the oracle: both heights and the sizes around them, more chains than
the table of low tiles holds, ragged last tiles, every tile width, with and
without a graph, the persistent schedule in between, and a workspace that holds
exactly what the batch asks for."""
import math

import numpy as np
import pytest
import torch

import oracle
import paper_1105_5804_gb300 as sw

pytestmark = pytest.mark.gpu

BATCHES = {
    "few": [64, 100, 260, 8], "rows8_last": [128] * 19, "rows16": [512, 300, 500, 516, 44], "rows32": [768, 1000, 900],
    "chains256": [4] * 256, "chains257": [8] * 257,
}


def _run(L, tile_w, graph, schedules):
    n = len(L)
    q = [2 + r % 3 if r % 5 else 9 for r in range(n)]
    beta = [0.8 * math.log(1 + math.sqrt(x)) for x in q]
    seed = [77 + r for r in range(n)]
    need = sw.sw_batch_device_bytes(L, q, tile_w=tile_w)
    ws = torch.full((need + 256,), 0x5A, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()   # the batch sets the workspace up on its own stream
    b = sw.sw_batch_create_ws(L, q, beta, seed, ws[:need], sw.SW_CONV_POTTS, True, 0, tile_w)
    try:
        sw.sw_batch_set_graph(b, graph)
        done = 0
        for schedule, k in schedules:
            sw.sw_batch_set_schedule(b, schedule)
            sw.sw_batch_sweep(b, k)
            done += k
        sw.sw_batch_sync(b)
        for r in range(0, n, max(1, n // 8)):
            T = oracle.threshold(beta[r])
            s, obs = oracle.chain(L[r], q[r], T, seed[r], 0, done, oracle.init_spins(L[r], q[r], seed[r], True))
            assert np.array_equal(sw.sw_batch_get_spins(b, r, L[r]), s), r
            assert np.array_equal(sw.sw_batch_observables(b, r, q[r]), obs), r
        assert bool((ws[need:] == 0x5A).all())
    finally:
        sw.sw_batch_destroy(b)


@pytest.mark.parametrize("name", list(BATCHES))
@pytest.mark.parametrize("graph", [False, True])
def test_chains(name, graph):
    _run(BATCHES[name], 256, graph, [(sw.SW_BATCH_PHASES, 3)])


@pytest.mark.parametrize("tile_w", sw.TILE_WIDTHS)
def test_widths_and_schedules(tile_w):
    P, Q = sw.SW_BATCH_PHASES, sw.SW_BATCH_PERSISTENT
    _run([36, 200, 324, 132], tile_w, True, [(P, 2), (Q, 2), (P, 1)])
