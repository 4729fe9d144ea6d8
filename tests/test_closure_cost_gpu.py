"""The closure and the residual of an iteration (kgs_close_sums) take time in
proportion to the cells: eight times the cells in at most twice eight times
the time (work that grew with their square took over twenty times as long).
The rescale keeps the total mass at every size.
"""
import time

import numpy as np
import pytest

from paper_1810_00348_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kgs():
    from paper_1810_00348_gb300 import kgs as k
    k.load()
    return k


def close_time(kgs, cells):
    import torch

    p = inputs.cavity(cells, 2, Kn=0.5)
    c = kgs.kgs_setup(p, precision=kgs.KGS_MIXED)
    sums = torch.empty(19 * p.ncell, dtype=torch.float64, device="cuda")
    kgs.kgs_sweep_sums(c, sums.data_ptr())
    torch.cuda.synchronize()
    best = float("inf")
    for _ in range(6):
        t0 = time.perf_counter()
        rc, _ = kgs.kgs_close_sums(c, sums.data_ptr())
        best = min(best, time.perf_counter() - t0)
        assert rc == kgs.KGS_OK
    rho = kgs.kgs_moments(c)[0]
    cell = p.dx[0] * p.dy[0] * p.dz[0]
    kgs.kgs_destroy(c)
    # the mass to keep is that of the uniform initial state, added cell by cell
    M0 = np.cumsum(np.full(p.ncell, cell))[-1]
    assert abs(float(np.sum(rho)) * cell - M0) <= 1e-13 * np.log2(p.ncell)
    return best


@pytest.mark.parametrize("cells", [[1, 1, 1], [31, 1, 1], [33, 3, 5], [8, 8, 128], [129, 64, 33]])
def test_rescale_keeps_the_mass(kgs, cells):
    close_time(kgs, cells)


def test_time_in_proportion_to_the_cells(kgs):
    small, large = close_time(kgs, [128, 128, 128]), close_time(kgs, [256, 256, 256])
    assert large <= 16.0 * small, "%.3g ms and %.3g ms" % (small * 1e3, large * 1e3)
