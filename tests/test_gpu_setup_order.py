"""A context's setup runs on its own stream, which does not wait for the legacy default
stream: its uploads and clears must be in that stream's order, whatever other work the
program has queued on the default stream meanwhile."""
import os
import threading

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


# one tile; resident tiles with vacuum around them; the solve's vectors in memory (uploads of
# 4 KB to 1 MB); each with the FP64 and the float-pair state
GRIDS = [(4, 4, 8), (9, 11, 13), (60, 58, 61)]


def _march(mot, grid, precision):
    eps = wl.sphere(max(grid), 12.0)[:grid[0], :grid[1], :grid[2]].copy()
    E = np.random.default_rng(1).normal(size=(6, eps.size, 3))
    E *= ((eps - 1.0) / eps).reshape(-1)[None, :, None]
    with mot.Context(eps, wl.fir_taps("fir3", 1e-3), precision=precision, scheme="blocked",
                     block=4) as own, own.share() as other:
        out = []
        for c in (own, other):
            c.set_excitation(E)
            out.append(c.march(6))
        return out


@pytest.mark.parametrize("precision", ["fp64", "fp32_history"])
@pytest.mark.parametrize("grid", GRIDS)
def test_creation_beside_work_on_the_default_stream(mot, grid, precision):
    """Contexts (one of its own setup, one that borrows it) created and marched while another
    thread keeps the default stream busy: the same bits as on an idle device."""
    torch = pytest.importorskip("torch")
    want = _march(mot, grid, precision)
    assert np.array_equal(want[0], want[1])
    a = torch.randn(4096, 4096, device="cuda")
    stop = threading.Event()

    def load():
        while not stop.is_set():
            for _ in range(8):
                torch.mm(a, a)
            torch.cuda.default_stream().synchronize()

    t = threading.Thread(target=load)
    t.start()
    try:
        for _ in range(3):
            for got in _march(mot, grid, precision):
                assert np.array_equal(got, want[0])
    finally:
        stop.set()
        t.join()
