"""GPU parity of the one-block kernel at the sizes where its parts change: the
last lattice on units of 8 rows and the first on units of 16 (80, 84), whole and
ragged units of 16 rows, the largest lattice it takes (112) and the first that
goes to the tiled kernels (116); degenerate thresholds, dense contacts and
switches to the tiled kernels on units of 16 rows."""
import math

import numpy as np
import pytest

import oracle
import paper_1105_5804_gb300 as sw

pytestmark = pytest.mark.gpu

SIZES = [76, 80, 84, 92, 96, 108, 112, 116]


def _check(h, L, q, T, seed, done, n, s):
    s, obs = oracle.chain(L, q, T, seed, done, n, s)
    assert np.array_equal(sw.sw_get_spins(h), s), (L, q, done, n)
    assert np.array_equal(sw.sw_observables(h, 4096), obs), (L, q, done, n)
    return s


@pytest.mark.parametrize("L", SIZES)
@pytest.mark.parametrize("q", [2, 3, 8, 9, 127])
def test_chains(L, q):
    T, seed = oracle.threshold(math.log(1 + math.sqrt(q))), 11 * L + q
    h = sw.sw_create_threshold(L, q, T, seed, True)
    try:
        s, done = oracle.init_spins(L, q, seed, True), 0
        for n in (1, 7, 2):
            sw.sw_sweep(h, n)
            s = _check(h, L, q, T, seed, done, n, s)
            done += n
    finally:
        sw.sw_destroy(h)


@pytest.mark.parametrize("L", [80, 84, 96, 112])
@pytest.mark.parametrize("q", [2, 9])
@pytest.mark.parametrize("T", [0, 1, 1 << 31, 3 << 30, (1 << 32) - 1, 1 << 32])
def test_thresholds(L, q, T):
    h = sw.sw_create_threshold(L, q, T, 5, True)
    try:
        sw.sw_sweep(h, 3)
        _check(h, L, q, T, 5, 0, 3, oracle.init_spins(L, q, 5, True))
    finally:
        sw.sw_destroy(h)


@pytest.mark.parametrize("L", [80, 96, 112])
@pytest.mark.parametrize("kind", ["rungs", "combs", "equal", "stairs"])
@pytest.mark.parametrize("T", [3 << 30, 1 << 32])
def test_dense_contacts(L, kind, T):
    """Spins whose runs touch as many runs of the row below as there can be:
    rows of one state and rows of alternating states, teeth of two sites, one
    state, and steps."""
    y, x = np.mgrid[0:L, 0:L]
    s = {"rungs": (y % 2) * (x % 2), "combs": (y % 2) * (x // 2 % 2), "equal": 0 * x, "stairs": (x + y) // 2 % 2}[kind]
    s = s.astype(np.int8).reshape(-1)
    h = sw.sw_create_threshold(L, 2, T, 9, False)
    try:
        sw.sw_set_spins(h, s)
        sw.sw_sweep(h, 2)
        _check(h, L, 2, T, 9, 0, 2, s)
    finally:
        sw.sw_destroy(h)


@pytest.mark.parametrize("L", [96, 112])
def test_switches(L):
    """Timing and the staged mode run the same chain on other kernels."""
    q, seed = 3, 17
    T = oracle.threshold(math.log(1 + math.sqrt(q)))
    h = sw.sw_create_threshold(L, q, T, seed, True)
    try:
        s, done = oracle.init_spins(L, q, seed, True), 0
        for step in ("plain", "timed", "plain", "staged", "plain"):
            sw.sw_set_timing(h, step == "timed")
            sw.sw_set_mode(h, sw.SW_MODE_STAGED if step == "staged" else sw.SW_MODE_FUSED)
            sw.sw_sweep(h, 2)
            s = _check(h, L, q, T, seed, done, 2, s)
            done += 2
    finally:
        sw.sw_destroy(h)
