"""GPU parity of the simple-cubic sweep in boxes whose last layer of bricks is
flat (its rows' draws are spread over the lanes by another rule, and only its
rows are swept) and in the boxes around them: every number of planes up to one
more than a brick's, second layers of 1 to 9, ragged rows and planes."""
import numpy as np
import pytest

import oracle
import paper_1105_5804_gb300 as sw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Z", list(range(1, 18)) + [18, 20, 23, 24, 25])
@pytest.mark.parametrize("X,Y", [(33, 9), (64, 16), (20, 3), (95, 17)])
@pytest.mark.parametrize("q,T", [(2, None), (9, None), (3, 3 << 30), (2, 0), (2, 1 << 32)])
def test_chain(X, Y, Z, q, T):
    T = oracle.threshold(0.4433 if q == 2 else 0.6) if T is None else T
    h = sw.sw3_create(X, Y, Z, q, T, 100 + Z, True)
    try:
        sw.sw3_sweep(h, 2)
        s, obs = oracle.chain3(X, Y, Z, q, T, 100 + Z, 0, 2, oracle.init_spins3(X, Y, Z, q, 100 + Z, True))
        assert np.array_equal(sw.sw3_get_spins(h), s)
        assert np.array_equal(sw.sw3_observables(h, 4096), obs)
    finally:
        sw.sw3_destroy(h)
