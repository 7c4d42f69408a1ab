"""The per-step solve on the shapes where its launch changes: one and several tiles of
8 x 4 x 4, ragged tiles, vacuum inside the tiles, grids with more tiles than resident
blocks, and 8^3 tiles; smooth and abrupt excitation (the fitted start, the extrapolated
start, a start worse than none).

The check is the defining equation itself: Z_0 J_n = E_n - P_{n-1} with Z_0 applied in
numpy from the table's lag-0 elements and P from mot_eval_history, which runs the march's
own history path on the same currents (so the history's rounding cancels)."""
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


def _z0_over_chi(ctx, eps, taps, J):
    """diag(1/chi) Z_0 J on the voxels with chi > 0 (zero elsewhere), J [M][3]."""
    W, V, U = eps.shape
    G = np.zeros((6, 2, 2, 2))
    tab = ctx.table(0, 1)[0]
    G[:, :min(W, 2), :min(V, 2), :min(U, 2)] = tab[:, :2, :2, :2]
    chi = (eps - 1.0) / eps
    act = chi > 0
    d0 = taps[0] if len(taps) else 0.0
    x = J.reshape(W, V, U, 3) * act[..., None]
    safe = np.where(act, chi, 1.0)
    out = x * ((0.5 / eps + d0) / safe)[..., None]
    pad = np.zeros((W + 2, V + 2, U + 2, 3))
    pad[1:-1, 1:-1, 1:-1] = x
    comp = {(0, 0): 0, (1, 1): 1, (2, 2): 2, (0, 1): 3, (0, 2): 4, (1, 2): 5}
    for ez in (-1, 0, 1):
        for ey in (-1, 0, 1):
            for ex in (-1, 0, 1):
                s = pad[1 + ez:1 + ez + W, 1 + ey:1 + ey + V, 1 + ex:1 + ex + U]
                e = (ex, ey, ez)
                for a in range(3):
                    for b in range(3):
                        g = G[comp[min(a, b), max(a, b)], abs(ez), abs(ey), abs(ex)]
                        if a != b:
                            g = g * np.sign(e[a]) * np.sign(e[b])
                        out[..., a] -= g * s[..., b]
    return (out * act[..., None]).reshape(-1, 3)


def _shape(kind, W, V, U):
    if kind == "cube":
        return np.full((W, V, U), 6.0)
    if kind == "holes":          # vacuum columns and a missing corner inside the tiles
        eps = np.full((W, V, U), 4.0)
        eps[:, ::3, ::2] = 1.0
        eps[W // 2:, V // 2:, U // 2:] = 1.0
        return eps
    z, y, x = ((np.arange(n) + 0.5 - n / 2.0) ** 2 / (n / 2.0) ** 2 for n in (W, V, U))
    return np.where(z[:, None, None] + y[None, :, None] + x[None, None, :] < 1.0, 12.0, 1.0)


# (grid, shape): one tile; one voxel beyond a tile on every axis; thin; ragged with holes;
# more 8 x 4 x 4 tiles than resident blocks; 8^3 tiles
CASES = [((4, 4, 8), "cube"), ((5, 5, 9), "cube"), ((2, 3, 17), "cube"), ((13, 9, 11), "holes"),
         ((26, 25, 31), "sphere"), ((46, 43, 50), "cube"), ((60, 58, 61), "holes")]


@pytest.mark.parametrize("precision,tol", [("fp64", 2e-13), ("fp32_history", 3.3e-8)])
@pytest.mark.parametrize("grid,kind", CASES)
def test_solution_satisfies_its_equation(mot, grid, kind, precision, tol):
    """tol: the solver's own tolerance (1e-13 / 3e-8 of ||b||, b = rhs / chi) with the
    rounding of this check's numpy sums (FP64) or a tenth (FP32-history)."""
    if precision == "fp64" and grid[0] > 50:
        grid = (33, 42, 50)                      # FP64 history of the largest grid is slow
    W, V, U = grid
    eps = _shape(kind, W, V, U)
    taps = wl.fir_taps("fir3", 1e-3)
    rng = np.random.default_rng(W + V + U)
    M = eps.size
    chi = ((eps - 1.0) / eps).reshape(-1)
    n = 12
    # smooth rise for six steps, nothing for two, then an unrelated field 1e4 times larger
    amp = [0.1, 0.3, 0.6, 0.8, 0.9, 1.0, 0.0, 0.0, 1e4, 9e3, 1e3, 1e1]
    f1, f2 = rng.normal(size=(2, M, 3)) * chi[:, None]
    E = np.stack([a * (f1 if i < 8 else f2) for i, a in enumerate(amp)])
    with mot.Context(eps, taps, precision=precision) as ctx:
        ctx.set_excitation(E)
        J = ctx.march(n)
        for i in (0, 3, 5, 7, 8, 11):
            P = ctx.eval_history(J[:i][::-1][:ctx.ell].copy()) if i else np.zeros((M, 3))
            b = (E[i] - P) * np.where(chi > 0, 1.0 / np.where(chi > 0, chi, 1.0), 0.0)[:, None]
            r = b - _z0_over_chi(ctx, eps, taps, J[i])
            assert np.linalg.norm(r) <= tol * np.linalg.norm(b), (i, np.linalg.norm(r) / np.linalg.norm(b))


@pytest.mark.parametrize("precision", ["fp64", "fp32_history"])
@pytest.mark.parametrize("grid,kind", [((5, 6, 40), "cube"), ((20, 21, 23), "holes")])
def test_repeated_marches_are_bitwise_equal(mot, grid, kind, precision):
    """Blocks of the solve run unordered between their exchanges; every sum is taken in a
    fixed order, so a march from rest gives the same bits every time."""
    W, V, U = grid
    eps = _shape(kind, W, V, U)
    rng = np.random.default_rng(5)
    E = rng.normal(size=(24, eps.size, 3)) * ((eps - 1.0) / eps).reshape(-1)[None, :, None]
    with mot.Context(eps, wl.fir_taps("fir3", 1e-3), precision=precision, scheme="blocked",
                     block=4) as ctx:
        first = None
        for _ in range(12):
            ctx.restart(0, None)
            ctx.set_excitation(E)
            J = ctx.march(24)
            first = J if first is None else first
            assert np.array_equal(J, first)
