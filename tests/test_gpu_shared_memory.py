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


# longest lengths that the general FFT tile takes (756 in FP64, 800 in FP32) and the next ones
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("precision,side,ok", [("fp64", 378, True), ("fp64", 383, False),
                                               ("fp32_history", 400, True),
                                               ("fp32_history", 404, False)])
def test_longest_transforms(mot, precision, side, ok, axis):
    """A length without a tile is refused at the first step of a march, on any axis and whichever
    kernels the other steps would take; the longest one marches (against a longer padding of the
    short axes, 1e-12 / 1e-5)."""
    grid = [2, 2, 2]
    grid[axis] = side
    eps = 2.0 + np.random.default_rng(2).random(grid)
    E = np.random.default_rng(3).normal(size=(5, eps.size, 3))

    def march(**kw):
        with mot.Context(eps, wl.fir_taps("fir3", 1e-3), precision=precision, **kw) as c:
            c.set_excitation(E)
            return c.march(5), tuple(c.P)

    for kw in (dict(scheme="direct"), dict(scheme="blocked", block=8)):
        if not ok:
            with pytest.raises(mot.MotError, match="MOT_ERR_ARG"):
                march(**kw)
            continue
        J, P = march(**kw)
        other, _ = march(fft_len=tuple(2 * p if p < 8 else p for p in P), **kw)
        tol = 1e-12 if precision == "fp64" else 1e-5
        assert np.linalg.norm(J - other) <= tol * np.linalg.norm(J)
