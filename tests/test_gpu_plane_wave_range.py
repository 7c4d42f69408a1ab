"""The tested plane wave at pulse centres and directions that leave no usable table."""
import os

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mot():
    from paper_2407_03323_gb300 import build, mot as m
    if not os.path.exists(m.LIB_PATH):
        build.build()
    m.load_library()
    return m


@pytest.mark.parametrize("t0", [1e6, 2.0 ** 40, 2.0 ** 44 / 9 - 1, 2.0 ** 44 / 9 + 1e3, 1e15, 1e17,
                                1e18, 1e300, np.inf, np.nan])
def test_far_and_non_finite_pulse_centres(mot, t0):
    """A pulse that far away is exactly zero (exp underflows); an infinite or undefined centre
    gives NaN on the scatterer; vacuum stays zero.  Steps in pieces of the table and one."""
    w = wl.pulse(9, 6.0)
    eps = np.full((5, 4, 9), 3.0)
    eps[0, 0, 0] = 1.0
    with mot.Context(eps) as c:
        for first, n in ((1, 1), (1, 33), (2 ** 30, 33)):
            for sign in (1.0, -1.0):
                E = np.asarray(c.plane_wave(w["k_hat"], w["p_hat"], w["f_c"], w["sigma_t"],
                                            sign * t0, first, n))
                assert (E[:, 0] == 0).all()
                assert np.isnan(E[:, 1:]).all() if not np.isfinite(t0) else (E[:, 1:] == 0).all()


def test_directions_without_a_table(mot):
    """r . k_hat far beyond the table (a direction that is not a unit vector), or none."""
    with mot.Context(np.full((3, 3, 3), 2.0)) as c:
        for k in ((0.0, 0.0, 1e6), (1e15, 0.0, 0.0), (0.0, -1e300, 0.0)):
            E = np.asarray(c.plane_wave(k, (1, 0, 0), 0.05, 10.0, 30.0, 1, 40))
            assert (E == 0).all()
        E = np.asarray(c.plane_wave((np.nan, 0, 0), (1, 1, 1), 0.05, 10.0, 30.0, 1, 40))
        assert np.isnan(E).all()
