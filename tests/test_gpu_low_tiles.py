"""GPU parity of fused sweeps on tiles of 8 and 16 rows (lattices with few
tiles) against the oracle: spins and the observables of every sweep, at the
edges of the ranges of both heights, for last tiles of full and ragged height
and width, state counts in registers and in the histogram, degenerate
thresholds, and the few-cluster update."""
import math

import numpy as np
import pytest

import oracle
import paper_1105_5804_gb300 as sw

pytestmark = pytest.mark.gpu

# 256-wide tiles: 8 rows up to L = 768 (304 tiles at most), 16 rows up to 1280
# (456), 32 rows above
SIZES = [132, 196, 256, 260, 512, 516, 764, 768, 772, 1000, 1024, 1028, 1280, 1284]


def _T(q):
    return oracle.threshold(math.log(1 + math.sqrt(q)))


def _check(h, L, q, T, seed, done, n, s):
    s, obs = oracle.chain(L, q, T, seed, done, n, s)
    assert np.array_equal(sw.sw_get_spins(h), s), (L, q, done, n)
    assert np.array_equal(sw.sw_observables(h, 4096), obs), (L, q, done, n)
    return s


@pytest.mark.parametrize("L", SIZES)
@pytest.mark.parametrize("q", [2, 3, 9])
def test_chains(L, q):
    T, seed = _T(q), 7 + L + q
    h = sw.sw_create_threshold(L, q, T, seed, True)
    try:
        s, done = oracle.init_spins(L, q, seed, True), 0
        for n in (1, 5):
            sw.sw_sweep(h, n)
            s = _check(h, L, q, T, seed, done, n, s)
            done += n
    finally:
        sw.sw_destroy(h)


@pytest.mark.parametrize("L", [132, 268, 900])
@pytest.mark.parametrize("T", [0, 1, 3 << 30, (1 << 32) - 1, 1 << 32])
def test_thresholds(L, T):
    h = sw.sw_create_threshold(L, 2, T, 5, False)
    try:
        s = oracle.init_spins(L, 2, 5, False)
        sw.sw_sweep(h, 3)
        _check(h, L, 2, T, 5, 0, 3, s)
    finally:
        sw.sw_destroy(h)


@pytest.mark.parametrize("L", [20, 132, 1004, 1300])
def test_few(L):
    q, T, P, seed = 3, _T(3), sw.sw_prob_threshold(0.5), 11
    h = sw.sw_create_threshold(L, q, T, seed, True)
    try:
        sw.sw_set_update(h, sw.SW_UPDATE_FEW, 4, P)
        sw.sw_sweep(h, 3)
        s, obs = oracle.few_chain(L, q, T, P, 4, seed, 0, 3, oracle.init_spins(L, q, seed, True))
        assert np.array_equal(sw.sw_get_spins(h), s)
        assert np.array_equal(sw.sw_observables(h, 4096), obs)
    finally:
        sw.sw_destroy(h)
