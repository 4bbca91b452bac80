"""GPU parity of the simple-cubic sweep's row loads, joins and merge against the
oracle: rows that start at every offset from an aligned word, last bricks of
every kind of width, both halves of a row ragged, boxes one brick long along
some axes, and state counts in registers and in the histogram."""
import numpy as np
import pytest

import oracle
import paper_1105_5804_gb300 as sw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("X", [1, 2, 3, 5, 15, 16, 17, 19, 31, 32, 33, 34, 46, 47, 48, 49, 64, 65, 79, 80, 100])
@pytest.mark.parametrize("Y,Z,q", [(7, 16, 2), (9, 5, 3), (19, 34, 9)])
def test_chains(X, Y, Z, q):
    T, seed = oracle.threshold(0.4433) if q == 2 else oracle.threshold(0.6), 100 + X
    h = sw.sw3_create(X, Y, Z, q, T, seed, True)
    try:
        sw.sw3_sweep(h, 3)
        s, obs = oracle.chain3(X, Y, Z, q, T, seed, 0, 3, oracle.init_spins3(X, Y, Z, q, seed, True))
        assert np.array_equal(sw.sw3_get_spins(h), s)
        assert np.array_equal(sw.sw3_observables(h, 4096), obs)
    finally:
        sw.sw3_destroy(h)


def test_all_bonds_open():
    """Every contact list at its fullest."""
    h = sw.sw3_create(96, 24, 48, 2, 1 << 32, 3, False)
    try:
        sw.sw3_sweep(h, 1)
        assert np.array_equal(sw.sw3_labels(h), np.zeros(96 * 24 * 48, dtype=np.int32))
    finally:
        sw.sw3_destroy(h)


@pytest.mark.parametrize("seed", range(6))
def test_no_horizontal_runs(seed):
    """Spins in columns along y and z: only y and z bonds are open, so that a
    plane's list of y contacts overflows."""
    X, Y, Z, q = 64, 16, 32, 3
    s = np.broadcast_to(np.arange(X) % 3, (Z, Y, X)).astype(np.int8).reshape(-1).copy()
    T = 3 << 30
    h = sw.sw3_create(X, Y, Z, q, T, seed, False)
    try:
        sw.sw3_set_spins(h, s)
        sw.sw3_sweep(h, 1)
        ref, _, lab, _ = oracle.sweep3(X, Y, Z, q, T, seed, 0, s)
        assert np.array_equal(sw.sw3_labels(h), lab)
        assert np.array_equal(sw.sw3_get_spins(h), ref)
    finally:
        sw.sw3_destroy(h)
