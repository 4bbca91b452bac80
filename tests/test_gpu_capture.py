"""Sweeps on a stream that is being captured are refused (they would not be
counted), in every update and for every size class, and the handle goes on
afterwards as if they had not been asked for."""
import math

import numpy as np
import pytest
import torch

import oracle
import paper_1105_5804_gb300 as sw

pytestmark = pytest.mark.gpu


def _refused(call, stream):
    side = torch.cuda.CUDAGraph()
    x = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.graph(side, stream=stream):
        x += 1.0
        with pytest.raises(sw.SwcclError) as e:
            call()
    assert e.value.code == sw.SW_ERR_CUDA
    torch.cuda.synchronize()


@pytest.mark.parametrize("L", [16, 128, 132, 1000, 1500])
@pytest.mark.parametrize("few", [False, True])
@pytest.mark.parametrize("warm", [0, 2])
def test_square(L, few, warm):
    T, seed, st = oracle.threshold(math.log(1 + math.sqrt(2))), 21, torch.cuda.Stream()
    P = sw.sw_prob_threshold(0.5)
    h = sw.sw_create_threshold(L, 2, T, seed, True, st.cuda_stream)
    try:
        if few:
            sw.sw_set_update(h, sw.SW_UPDATE_FEW, 4, P)
        sw.sw_sweep(h, warm)
        _refused(lambda: sw.sw_sweep(h, 2), st)
        sw.sw_sweep(h, 1)
        s = oracle.init_spins(L, 2, seed, True)
        if few:
            s, obs = oracle.few_chain(L, 2, T, P, 4, seed, 0, warm + 1, s)
        else:
            s, obs = oracle.chain(L, 2, T, seed, 0, warm + 1, s)
        assert np.array_equal(sw.sw_get_spins(h), s)
        assert np.array_equal(sw.sw_observables(h, 4096), obs)
    finally:
        sw.sw_destroy(h)


@pytest.mark.parametrize("warm", [0, 2])
def test_cubic(warm):
    T, st = oracle.threshold(0.4433), torch.cuda.Stream()
    h = sw.sw3_create(33, 9, 17, 2, T, 4, True, st.cuda_stream)
    try:
        sw.sw3_sweep(h, warm)
        _refused(lambda: sw.sw3_sweep(h, 2), st)
        sw.sw3_sweep(h, 1)
        s, obs = oracle.chain3(33, 9, 17, 2, T, 4, 0, warm + 1, oracle.init_spins3(33, 9, 17, 2, 4, True))
        assert np.array_equal(sw.sw3_get_spins(h), s)
        assert np.array_equal(sw.sw3_observables(h, 4096), obs)
    finally:
        sw.sw3_destroy(h)
