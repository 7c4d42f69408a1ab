"""Launches near the limits of a block's shared memory."""
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


@pytest.mark.parametrize("k", [6135, 6136, 6143, 6144, 6150])
def test_long_lanczos(mot, k):
    """Reorthogonalised Lanczos on both sides of 48 KB of coefficients (k = 6143), on an operator
    of dimension 12: the recurrence ends with the subspace, at the spectrum that 12 steps give."""
    with mot.Context(np.array([[[2.0, 3.0], [4.0, 5.0]]])) as c:
        r = c.pdsa_lanczos(c.ell, k, seed=2, reorth=True, n_out=1)
        ref = c.pdsa_lanczos(c.ell, 12, seed=2, reorth=True, n_out=1)
        assert r["steps"] <= 13
        for a in ("theta_max", "ritz"):
            assert np.allclose(r[a], ref[a], rtol=1e-10, atol=0)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32_history", 1e-5)])
def test_level_of_256_lags(mot, precision, tol):
    """A level of length 256 (general kernel, static index lists beside its dynamic lines) against
    the direct sum: FP64 to 1e-12, FP32-history to 1e-5 of FP64."""
    eps = 2.0 + np.random.default_rng(0).random((1, 1, 260))
    n = 300
    E = np.random.default_rng(1).normal(size=(n, eps.size, 3))
    out = []
    for kw in (dict(precision="fp64", scheme="direct"),
               dict(precision=precision, scheme="blocked", block=256)):
        with mot.Context(eps, wl.fir_taps("fir3", 1e-3), **kw) as c:
            c.set_excitation(E)
            out.append(c.march(n))
    assert np.linalg.norm(out[1] - out[0]) <= tol * np.linalg.norm(out[0])
