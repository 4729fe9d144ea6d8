"""Waits that expire at any place of the persistent sweep (a limit of one or a
few polls) end the launch with KGS_ETIMEOUT in every kernel that uses them; the
batch then works as before, bit for bit.
"""
import numpy as np
import pytest

from paper_1810_00348_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kgs():
    from paper_1810_00348_gb300 import kgs as k
    k.load()
    return k


@pytest.mark.parametrize("precision,v_per_cta", [(0, 128), (1, 128), (1, 256)])
def test_short_limits_report_and_recover(kgs, precision, v_per_cta):
    probs = [inputs.cavity([19, 18, 9], [12, 11, 10], Kn=0.5), inputs.cavity([9, 26, 11], [32, 9, 8], Kn=0.3)]
    b = kgs.kgs_batch_setup(probs, precision=precision, v_per_cta=v_per_cta, block_z=4)
    rc, done, res = kgs.kgs_batch_iterate(b, 2)
    assert rc == kgs.KGS_OK and done == [2, 2]
    want = [kgs.kgs_batch_moments(b, i).copy() for i in range(2)]
    expired = 0
    for limit in (1, 1, 1, 2, 3, 10, 30):
        kgs.kgs_batch_fault(b, spin_limit=limit)
        for i in range(2):
            kgs.kgs_batch_set_initial(b, i)
        rc, _, _ = kgs.kgs_batch_iterate(b, 1)
        assert rc in (kgs.KGS_OK, kgs.KGS_ETIMEOUT)
        expired += rc == kgs.KGS_ETIMEOUT
    assert expired > 0  # a block takes microseconds, a poll 100 ns
    kgs.kgs_batch_fault(b)
    for i in range(2):
        kgs.kgs_batch_set_initial(b, i)
    assert kgs.kgs_batch_iterate(b, 2) == (kgs.KGS_OK, [2, 2], res)
    assert all(np.array_equal(kgs.kgs_batch_moments(b, i), want[i]) for i in range(2))
