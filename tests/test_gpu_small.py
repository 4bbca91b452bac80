"""GPU parity of the small-lattice kernel (many sweeps of a lattice up to 128
on a side per launch) against the oracle: spins and the observables of every
sweep, for units that are whole, ragged in one direction or both, and wrapped
onto themselves; more states than the register counters hold; degenerate
thresholds; more sweeps than one launch takes; and switches between this kernel
and the tiled one (timing, few-cluster update, staged mode, new spins)."""
import math

import numpy as np
import pytest

import oracle
import paper_1105_5804_gb300 as sw

pytestmark = pytest.mark.gpu


def _T(q):
    return oracle.threshold(math.log(1 + math.sqrt(q)))


def _check(h, L, q, T, seed, done, n, s):
    s, obs = oracle.chain(L, q, T, seed, done, n, s)
    assert np.array_equal(sw.sw_get_spins(h), s), (L, q, done, n)
    assert np.array_equal(sw.sw_observables(h, 4096), obs), (L, q, done, n)
    return s


@pytest.mark.parametrize("L", [4, 12, 16, 20, 32, 36, 60, 64, 100, 124, 128, 132])
@pytest.mark.parametrize("q", [2, 3, 8, 9, 127])
def test_chains(L, q):
    T, seed = _T(q), 40 + L + q
    h = sw.sw_create_threshold(L, q, T, seed, True)
    try:
        s, done = oracle.init_spins(L, q, seed, True), 0
        for n in (1, 2, 17, 1):
            sw.sw_sweep(h, n)
            s = _check(h, L, q, T, seed, done, n, s)
            done += n
    finally:
        sw.sw_destroy(h)


@pytest.mark.parametrize("L", [16, 36, 128])
@pytest.mark.parametrize("T", [0, 1, 3 << 30, (1 << 32) - 1, 1 << 32])
def test_thresholds(L, T):
    h = sw.sw_create_threshold(L, 3, T, 5, True)
    try:
        sw.sw_sweep(h, 6)
        _check(h, L, 3, T, 5, 0, 6, oracle.init_spins(L, 3, 5, True))
    finally:
        sw.sw_destroy(h)


def test_more_sweeps_than_a_launch():
    L, q, T, n = 8, 2, _T(2), 2500
    h = sw.sw_create_threshold(L, q, T, 3, True)
    try:
        sw.sw_sweep(h, n)
        _check(h, L, q, T, 3, 0, n, oracle.init_spins(L, q, 3, True))
    finally:
        sw.sw_destroy(h)


def test_switching_between_paths():
    """Observables left uncounted by one path are counted by the other."""
    L, q, T, seed = 68, 2, _T(2), 9
    h = sw.sw_create_threshold(L, q, T, seed, True)
    try:
        s, done, rows = oracle.init_spins(L, q, seed, True), 0, []
        for n, timing in ((3, False), (2, True), (4, False), (1, True), (1, False)):
            sw.sw_set_timing(h, timing)
            sw.sw_sweep(h, n)
            s, obs = oracle.chain(L, q, T, seed, done, n, s)
            rows.append(obs)
            done += n
        sw.sw_set_timing(h, False)
        assert np.array_equal(sw.sw_observables(h, 4096), np.concatenate(rows))
        assert np.array_equal(sw.sw_get_spins(h), s)
        P = sw.sw_prob_threshold(0.5)
        sw.sw_set_update(h, sw.SW_UPDATE_FEW, 4, P)
        sw.sw_sweep(h, 2)
        s, few = oracle.few_chain(L, q, T, P, 4, seed, done, 2, s)
        done += 2
        sw.sw_set_update(h, sw.SW_UPDATE_SW)
        sw.sw_sweep(h, 3)
        s, obs = oracle.chain(L, q, T, seed, done, 3, s)
        done += 3
        assert np.array_equal(sw.sw_observables(h, 4096), np.concatenate([few, obs]))
        sw.sw_set_mode(h, sw.SW_MODE_STAGED)
        sw.sw_sweep(h, 1)
        s = _check(h, L, q, T, seed, done, 1, s)
        done += 1
        sw.sw_set_mode(h, sw.SW_MODE_FUSED)
        s = np.roll(s, 7)
        sw.sw_set_spins(h, s)
        sw.sw_sweep(h, 2)
        _check(h, L, q, T, seed, done, 2, s)
    finally:
        sw.sw_destroy(h)
