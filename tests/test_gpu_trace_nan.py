"""The traceback never takes a NaN value for the largest (a search compares each value with the
best one before it), except as the first state, which stays the best of none."""
import numpy as np
import pytest

import paper_2008_06888_gb300 as P

pytestmark = pytest.mark.gpu
INF, NAN = np.inf, np.nan


# values of the states ++, +-, -+, -- of two spins with a bond J and a field h on the first
@pytest.mark.parametrize("J,h,E", [(INF, INF, -INF),     # inf, NaN, -inf, NaN
                                   (INF, -INF, -INF),    # NaN, -inf, NaN, inf
                                   (NAN, 0.0, NAN)])     # NaN all
def test_two_spins(J, h, E):
    sg = P.SpinGlass(dict(n=2, q=2, edges=np.array([[0, 1]], np.int32),
                          J=np.array([0.5], np.float32), h=np.array([0.5, 0], np.float32)),
                     order="sweep", seq=np.arange(2, dtype=np.int32))
    try:
        got, s = sg.config_batch(np.array([[J]], np.float32), np.array([[h, 0]], np.float32))
        assert np.array_equal(got, [E], equal_nan=True) and s.tolist() == [[1, 1]]
    finally:
        sg.close()
