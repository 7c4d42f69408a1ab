"""The batched driver's memory estimate against what a march state takes on the device."""
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


# small grid, the driver's largest sides, a block beyond every lag (no accumulators, so that the
# estimate has no slack from the doubling plan), 9 taps (a longer J ring)
@pytest.mark.parametrize("precision", ["fp64", "fp32_history"])
@pytest.mark.parametrize("N,block,taps", [(16, 8, "fir3"), (48, 8, "fir3"), (48, 128, "fir3"),
                                          (64, 128, "binom9")])
def test_estimate_covers_a_march_state(mot, N, block, taps, precision):
    """Device memory taken by a context that borrows another's setup (its state and nothing
    else): covered by the estimate, up to the allocator's 2 MB pages of about 20 buffers."""
    torch = pytest.importorskip("torch")
    from paper_2407_03323_gb300.batch import march_bytes
    t = wl.fir_taps(taps, 1e-3)
    with mot.Context(np.full((N, N, N), 4.0), t, precision=precision, scheme="blocked",
                     block=block) as c:
        with c.share():
            pass
        free = torch.cuda.mem_get_info()[0]
        with c.share():
            used = free - torch.cuda.mem_get_info()[0]
    est = march_bytes(N, precision, block, n_taps=len(t))
    assert used <= est + 20 * (2 << 20)
    assert est <= 1.5 * used + 20 * (2 << 20)
