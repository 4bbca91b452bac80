"""Labeling calls recorded into a caller's graph, behind work of the caller on
the same stream and on a second one that is joined, and replayed on other
inputs: their programmatic launches wait for all of it, in every tile height."""
import numpy as np
import pytest
import torch

import oracle
import paper_1105_5804_gb300 as sw

pytestmark = pytest.mark.gpu

SHAPES = [(37, 130), (200, 300), (900, 1000), (1400, 1501)]


@pytest.mark.parametrize("H,W", SHAPES)
@pytest.mark.parametrize("call", ["label", "ws", "noalloc", "batch"])
def test_replays(H, W, call):
    side, main = torch.cuda.Stream(), torch.cuda.Stream()
    a, b = (torch.zeros(H * W, dtype=torch.uint8, device="cuda") for _ in range(2))
    px = torch.zeros(H * W, dtype=torch.uint8, device="cuda")
    half = torch.zeros(H * W, dtype=torch.uint8, device="cuda")
    mask = torch.zeros(sw.mask_bytes(H * W), dtype=torch.uint8, device="cuda")
    lab = torch.zeros(H * W, dtype=torch.int32, device="cuda")
    out = torch.zeros(H * W, dtype=torch.int32, device="cuda")
    ws = torch.empty(max(sw.ccl_workspace_bytes(H, W), sw.ccl_batch_workspace_bytes([H], [W])), dtype=torch.uint8,
                     device="cuda")
    label = {"label": lambda: sw.ccl_label(mask, lab, H, W, True, main),
             "ws": lambda: sw.ccl_label_ws(mask, lab, H, W, True, ws, main),
             "noalloc": lambda: sw.ccl_label_noalloc(mask, lab, H, W, True, main),
             "batch": lambda: sw.ccl_label_batch([mask], [lab], [H], [W], [True], ws, main)}[call]
    label()   # the first call on a device sets up what later ones find
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=main):
        side.wait_stream(main)
        with torch.cuda.stream(side):
            torch.bitwise_and(b, 1, out=half)
        torch.bitwise_and(a, 3, out=px)
        main.wait_stream(side)
        sw.ccl_bonds_from_pixels(px, mask, H, W, True, main)
        label()
        torch.add(lab, 1, out=out)
        main.wait_stream(side)
        px.bitwise_xor_(half)
        sw.ccl_bonds_from_pixels(px, mask, H, W, True, main)
        label()
    rng = np.random.default_rng(H)
    for _ in range(3):
        av, bv = (rng.integers(0, 3, H * W).astype(np.uint8) for _ in range(2))
        a.copy_(torch.from_numpy(av))
        b.copy_(torch.from_numpy(bv))
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        sw.ccl_status()
        first = oracle.label(oracle.bonds_from_pixels((av & 3).reshape(H, W), True), H, W, True)[0]
        second = oracle.label(oracle.bonds_from_pixels(((av & 3) ^ (bv & 1)).reshape(H, W), True), H, W, True)[0]
        assert np.array_equal(out.cpu().numpy(), first + 1)
        assert np.array_equal(lab.cpu().numpy(), second)


def test_a_batch_sweep_replayed_once():
    """Direct launches in a caller's graph: the sweeps count when they are
    recorded, and are read after one launch of the graph."""
    L, q, beta, seed = [64, 300], [2, 3], [0.44, 1.0], [5, 6]
    st = torch.cuda.Stream()
    b = sw.sw_batch_create(L, q, beta, seed, sw.SW_CONV_AUTO, True, st.cuda_stream)
    try:
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            sw.sw_batch_sweep(b, 3)
        g.replay()
        torch.cuda.synchronize()
        sw.sw_batch_sweep(b, 2)
        for r in range(2):
            T = sw.sw_threshold_for(q[r], beta[r], 1.0, sw.SW_CONV_AUTO)
            s, obs = oracle.chain(L[r], q[r], T, seed[r], 0, 5, oracle.init_spins(L[r], q[r], seed[r], True))
            assert np.array_equal(sw.sw_batch_get_spins(b, r, L[r]), s)
            assert np.array_equal(sw.sw_batch_observables(b, r, q[r]), obs)
    finally:
        sw.sw_batch_destroy(b)
