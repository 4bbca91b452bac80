"""GPU parity of the few-cluster flip against the oracle where its parts can go
wrong: rows whose selection bits straddle words, a seed on every site (the list
of roots takes several passes), one seed, clusters that always or never move,
the most states there are, and tiles that no selected cluster reaches."""
import math

import numpy as np
import pytest

import oracle
import paper_1105_5804_gb300 as sw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [4, 36, 260, 300, 1004, 1320, 1600])
@pytest.mark.parametrize("q,ratio", [(2, 1.0), (3, 0.3), (127, 1.0)])
@pytest.mark.parametrize("ell", ["one", "four", "all"])
@pytest.mark.parametrize("P", [0, 1 << 31, 1 << 32])
def test_few(L, q, ratio, ell, P):
    ell = {"one": 1, "four": 4, "all": L}[ell]
    T, seed = oracle.threshold(ratio * math.log(1 + math.sqrt(q))), 5 + L + q
    h = sw.sw_create_threshold(L, q, T, seed, True)
    try:
        sw.sw_set_update(h, sw.SW_UPDATE_FEW, ell, P)
        sw.sw_sweep(h, 2)
        s, obs = oracle.few_chain(L, q, T, P, ell, seed, 0, 2, oracle.init_spins(L, q, seed, True))
        assert np.array_equal(sw.sw_get_spins(h), s)
        assert np.array_equal(sw.sw_observables(h, 4096), obs)
    finally:
        sw.sw_destroy(h)
