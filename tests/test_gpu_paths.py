"""Dispatch edges of the march: the same problem through different kernels.

A march's result does not depend on the FFT lengths (any length >= 2N - 1 per axis), on the
scheme or on how the output leaves, but the kernels do: x and y passes in one kernel or two,
four-step codelets, fused z passes with 1 to 8 lines a block, levels on their own lengths."""
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


def _noise(grid, seed=0):
    rng = np.random.default_rng(seed + sum(grid))
    return 2.0 + 4.0 * rng.random(grid)


def _march(mot, eps, steps, **kw):
    n = max(eps.shape)
    w = wl.pulse(n, 6.0)
    with mot.Context(eps, wl.fir_taps("fir3", 1e-7 * n ** 3), **kw) as c:
        # (from 40 steps before the pulse's centre: every step matters)
        E = c.plane_wave(w["k_hat"], w["p_hat"], w["f_c"], w["sigma_t"], w["t0"] - 40, 1, steps)
        c.set_excitation(E)
        return c.march(steps), tuple(c.P)


# grid (W, V, U), FFT lengths (u, v, w) of the other route: one row pair per plane and an odd
# row; planes in one kernel against codelets; lines longer than the one-kernel rule takes;
# numbers of planes on both sides of FP64's rule (150, 153, 306); radices 5 and 7
ROUTES = [((1, 1, 3), (64, 96, 64)), ((2, 3, 5), (210, 210, 10)), ((7, 6, 9), (64, 64, 64)),
          ((5, 17, 33), (210, 96, 64)), ((50, 9, 20), (64, 64, 100)), ((51, 9, 20), (64, 64, 108)),
          ((102, 9, 20), (64, 64, 216)),
          ((4, 9, 70), (140, 28, 14)), ((9, 70, 4), (14, 140, 28))]


@pytest.mark.parametrize("grid,other", ROUTES)
def test_fft_routes_agree(mot, grid, other):
    """FP64 to 1e-12 (the rounding of two different transforms), FP32-history of either route
    to 1e-5 of the FP64 march."""
    eps = _noise(grid)
    kw = dict(scheme="blocked", block=4)
    ref, P0 = _march(mot, eps, 48, precision="fp64", **kw)
    got, P1 = _march(mot, eps, 48, precision="fp64", fft_len=other, **kw)
    assert P1 == other != P0
    nrm = np.linalg.norm(ref)
    assert np.linalg.norm(got - ref) <= 1e-12 * nrm
    for extra in ({}, {"fft_len": other}):
        f32, _ = _march(mot, eps, 48, precision="fp32_history", **kw, **extra)
        assert np.linalg.norm(f32 - ref) <= 1e-5 * nrm, extra


@pytest.mark.parametrize("grid", [(1, 2, 2), (4, 4, 3), (8, 9, 8), (16, 17, 18), (33, 24, 31)])
def test_schemes_agree(mot, grid):
    """Direct and blocked schemes (blocks 2 to 16: level lengths from 2 to the longest that
    fits) to 1e-12 in FP64 and 1e-5 in FP32-history."""
    eps = _noise(grid, 1)
    ref, _ = _march(mot, eps, 72, precision="fp64", scheme="direct")
    nrm = np.linalg.norm(ref)
    for precision, tol in (("fp64", 1e-12), ("fp32_history", 1e-5)):
        for block in (0, 2, 4, 8, 16):
            kw = dict(scheme="blocked", block=block) if block else dict(scheme="direct")
            got, _ = _march(mot, eps, 72, precision=precision, **kw)
            assert np.linalg.norm(got - ref) <= tol * nrm, (precision, block)


@pytest.mark.parametrize("precision", ["fp64", "fp32_history"])
@pytest.mark.parametrize("grid,corner", [((9, 10, 20), (2, 3, 4)), ((26, 27, 40), (26, 5, 9)),
                                         ((96, 8, 120), (90, 8, 100))])
def test_vacuum_outputs_and_norms(mot, grid, corner, precision):
    """Scatterer in a corner: voxels in none of the solve's tiles, vacuum voxels inside them
    (the last grid's solve keeps its vectors in memory).  With eps = 1 the equation is
    (1/2 + d_0) J_n = E_n - (1/2 + d_1) J_{n-1} - d_2 J_{n-2}, three FP64 terms: 1e-13.  Host
    and device outputs are the same bits, and the last norm is that of the last output."""
    torch = pytest.importorskip("torch")
    eps = np.ones(grid)
    eps[:corner[0], :corner[1], :corner[2]] = 5.0
    taps = wl.fir_taps("fir3", 1e-3)
    rng = np.random.default_rng(3)
    n = 9
    E = rng.normal(size=(n, eps.size, 3))
    vac = (eps == 1.0).reshape(-1)
    with mot.Context(eps, taps, precision=precision, scheme="blocked", block=4) as c:
        c.set_excitation(E)
        J = c.march(n)
        norm = c.info()["last_norm"]
        c.restart(0, None)
        c.set_excitation(torch.from_numpy(E).cuda())
        out = torch.full((n, eps.size, 3), np.nan, dtype=torch.float64, device="cuda")
        c.march(n - 1, out=out[:n - 1])
        c.march(1, out=out[n - 1:])
        assert c.info()["last_norm"] == norm
        assert np.array_equal(out.cpu().numpy(), J)
    assert abs(norm - np.linalg.norm(J[-1])) <= 1e-12 * norm
    d = list(taps) + [0.0] * 3
    want = np.zeros((n, int(vac.sum()), 3))
    for i in range(n):
        r = E[i][vac]
        if i > 0:
            r = r - (0.5 + d[1]) * want[i - 1]
        if i > 1:
            r = r - d[2] * want[i - 2]
        want[i] = r / (0.5 + d[0])
    assert np.abs(J[:, vac] - want).max() <= 1e-13 * np.abs(want).max()


@pytest.mark.parametrize("n0", [1, 40000])
def test_plane_wave_in_pieces(mot, n0):
    """Steps are dealt out 16 a thread from a call's first step: one call of 49 steps and calls
    of 1, 15, 16 and 17 give the same field, at step 40000 too (1e-14 of its largest value)."""
    grid = (5, 4, 7)
    w = wl.pulse(7, 6.0)
    with mot.Context(_noise(grid), wl.fir_taps("fir3", 1e-4)) as c:
        def wave(first, count):
            return np.asarray(c.plane_wave(w["k_hat"], w["p_hat"], w["f_c"], w["sigma_t"],
                                           n0 + 20.0, first, count))
        whole = wave(n0, 49)
        parts, at = [], n0
        for k in (1, 15, 16, 17):
            parts.append(wave(at, k))
            at += k
    assert np.abs(whole).max() > 0
    assert np.abs(np.concatenate(parts) - whole).max() <= 1e-14 * np.abs(whole).max()


def test_lanczos_across_reads(mot):
    """The scalars of the reorthogonalised Lanczos are read every 32 steps: with more steps the
    extreme Ritz values move outwards only (interlacing, to 1e-12 of the largest), on both
    sides of a read."""
    with mot.Context(_noise((4, 5, 6))) as c:
        last = None
        for k in (1, 2, 31, 32, 33, 64, 65):
            r = c.pdsa_lanczos(c.ell, k, seed=2, reorth=True, n_out=1)
            assert r["steps"] == k
            low, high = r["ritz"][0], r["theta_max"]
            if last:
                assert low <= last[0] + 1e-12 * high and high >= last[1] - 1e-12 * high
            last = (low, high)
