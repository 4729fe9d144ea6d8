"""Problems that fit the device only without the tables that make a sweep
faster: they are set up, tuned and run all the same.  The rest of the device
is held by a tensor meanwhile, which touches no memory.
"""
import contextlib

import numpy as np
import pytest

from paper_1810_00348_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kgs():
    from paper_1810_00348_gb300 import kgs as k
    k.load()
    return k


@contextlib.contextmanager
def leave(nbytes):
    """Leave about nbytes of device memory free."""
    import torch

    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    hog = torch.empty(free - int(nbytes), dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del hog
        torch.cuda.empty_cache()


MB = 1 << 20
CELLS = [62, 64, 63]  # 256 MB of accumulators, 375 MB of axis factors with 16^3 velocities


def sizes(kgs, p, **kw):
    """Device bytes of a context with all its tables, and of the axis factors."""
    c = kgs.kgs_setup(p, precision=kgs.KGS_FP64, **kw)
    n = kgs.kgs_info(c)["device_bytes"]
    kgs.kgs_destroy(c)
    return n, p.ncell * (len(p.xi_x) + len(p.xi_y) + len(p.xi_z)) * 32


def test_fp64_without_room_for_axis_factors(kgs):
    p = inputs.cavity(CELLS, 16, Kn=0.5)
    full, factors = sizes(kgs, p)
    assert factors > 300 * MB
    ref = kgs.kgs_setup(p, precision=kgs.KGS_FP64)
    assert kgs.kgs_iterate(ref, 1)[0] == kgs.KGS_OK
    want = kgs.kgs_moments(ref).copy()
    kgs.kgs_destroy(ref)
    with leave(full - 100 * MB):  # the factors fit, or what they leave no room for
        c = kgs.kgs_setup(p, precision=kgs.KGS_FP64)
        assert kgs.kgs_info(c)["device_bytes"] < full - 200 * MB
        assert kgs.kgs_iterate(c, 1)[0] == kgs.KGS_OK
        got = kgs.kgs_moments(c)
        kgs.kgs_destroy(c)
    assert np.max(np.abs(got - want)) <= 1e-12


def test_autotune_and_batch_without_room_for_axis_factors(kgs):
    p = inputs.cavity(CELLS, 16, Kn=0.4)
    full, _ = sizes(kgs, p)
    with leave(full - 100 * MB):
        vpc, bz = kgs.kgs_autotune(p, precision=kgs.KGS_FP64)
    assert vpc == 128 and bz in (8, 16, 32)
    q = inputs.cavity(CELLS, 16, Kn=0.3)  # not tuned yet: the batch tunes it
    with leave(full - 100 * MB):
        b = kgs.kgs_batch_setup([q], precision=kgs.KGS_FP64)
        rc, done, _ = kgs.kgs_batch_iterate(b, 1)
        assert rc == kgs.KGS_OK and done == [1]
        kgs.kgs_batch_destroy(b)


def test_batch_takes_its_device_memory_at_set_up(kgs):
    """The work list is there before the factors, not looked for at the first iteration."""
    import torch

    p = inputs.cavity([8, 8, 256], 24, Kn=0.5)
    b = kgs.kgs_batch_setup([p] * 8, precision=kgs.KGS_FP64, v_per_cta=128, block_z=1)
    before = torch.cuda.mem_get_info()[0]
    assert kgs.kgs_batch_iterate(b, 1)[0] == kgs.KGS_OK
    # 8 instances x 256 blocks x 112 groups, 20 bytes each: 4.6 MB, in two allocations of 2 MB pages
    taken = before - torch.cuda.mem_get_info()[0]
    kgs.kgs_batch_destroy(b)
    assert taken < 4 * MB, taken


def few_velocities():
    # one velocity group per octant: all eight octants share one accumulator of 128 bytes per cell, or use eight
    return inputs.cavity([96, 100, 92], 4, Kn=0.5)


@pytest.mark.parametrize("precision", [0, 1])
def test_context_and_batch_with_room_for_one_accumulator(kgs, precision):
    p = few_velocities()
    c = kgs.kgs_setup(p, precision=precision)
    full = kgs.kgs_info(c)["device_bytes"]
    assert kgs.kgs_iterate(c, 2)[0] == kgs.KGS_OK
    want = kgs.kgs_moments(c).copy()
    kgs.kgs_destroy(c)
    extra = 7 * 128 * p.ncell + (12 * 32 * p.ncell if precision == kgs.KGS_FP64 else 0)
    with leave(full - extra + 200 * MB):
        c = kgs.kgs_setup(p, precision=precision)
        assert kgs.kgs_iterate(c, 2)[0] == kgs.KGS_OK
        got = kgs.kgs_moments(c).copy()
        kgs.kgs_destroy(c)
        b = kgs.kgs_batch_setup([p], precision=precision, v_per_cta=0 if precision else 128, block_z=32)
        assert kgs.kgs_batch_iterate(b, 2)[0] == kgs.KGS_OK
        batch = kgs.kgs_batch_moments(b, 0).copy()
        kgs.kgs_batch_destroy(b)
    tol = 1e-12 if precision == kgs.KGS_FP64 else 1e-5
    assert np.max(np.abs(got - want)) <= tol and np.max(np.abs(batch - want)) <= tol


def test_solvers_hold_one_phase_at_a_time(kgs):
    p = few_velocities()
    c = kgs.kgs_setup(p, precision=kgs.KGS_FP64)
    full = kgs.kgs_info(c)["device_bytes"]
    kgs.kgs_destroy(c)
    # room for the FP64 phase with one accumulator and no axis factors
    with leave(full - (7 * 128 + 12 * 32) * p.ncell + 250 * MB):
        rc, m, nm, nd, r = kgs.kgs_solve(p, tol=0.9, max_iters=50)
        assert rc == kgs.KGS_OK and nd >= 1 and r < 0.9
        rc, b, nm, nd, res = kgs.kgs_batch_solve([p], tol=0.9, max_iters=50, v_per_cta=256, block_z=32)
        assert rc == kgs.KGS_OK and nd[0] >= 1 and res[0] < 0.9
        kgs.kgs_batch_destroy(b)


def test_tables_for_speed_take_a_third_of_free_memory_at_most(kgs):
    p = inputs.cavity(CELLS, 16, Kn=0.5)
    full, factors = sizes(kgs, p)
    held = {}
    for more in (0.5, 1.5, 2.5, 4.0):  # left free beside the context, in factors
        with leave(full + more * factors):
            c = kgs.kgs_setup(p, precision=kgs.KGS_FP64)
            held[more] = kgs.kgs_info(c)["device_bytes"]
            kgs.kgs_destroy(c)
            b = kgs.kgs_batch_setup([p], precision=kgs.KGS_FP64, v_per_cta=128, block_z=32)
            assert kgs.kgs_batch_info(b, 0)["device_bytes"] >= factors or more < 2.0
            kgs.kgs_batch_destroy(b)
    assert held[2.5] == held[4.0] == full
    assert held[0.5] == held[1.5] <= full - factors
    q = few_velocities()
    c = kgs.kgs_setup(q, precision=kgs.KGS_MIXED)
    full = kgs.kgs_info(c)["device_bytes"]
    kgs.kgs_destroy(c)
    with leave(full + 1.5 * 7 * 128 * q.ncell):
        c = kgs.kgs_setup(q, precision=kgs.KGS_MIXED)
        assert kgs.kgs_info(c)["device_bytes"] == full - 7 * 128 * q.ncell
        kgs.kgs_destroy(c)
