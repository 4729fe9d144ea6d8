"""Velocity x-lines longer than half a packed group (128 nodes per octant) that
groups cut anywhere, so that a half of a group can lie inside one line: both
precisions in a context, and the mixed one in a batch and through the entry
point without device allocation, against the FP64 oracle at the tolerances of
the parity tests (1e-10 and 1e-5).
"""
import numpy as np
import pytest

from oracle import Oracle
from paper_1810_00348_gb300 import inputs
from tests.parity import assert_fields_close, assert_rho_w_close

pytestmark = pytest.mark.gpu

FP64_TOL = 1e-10
MIXED_TOL = 1e-5


@pytest.fixture(scope="module")
def kgs():
    from paper_1810_00348_gb300 import kgs as k
    k.load()
    return k


@pytest.mark.parametrize("vels", [[300, 4, 6], [400, 2, 4], [266, 6, 4], [520, 2, 2]])
def test_groups_that_cut_long_lines(kgs, vels):
    import torch

    p = inputs.cavity([4, 9, 3], vels, L_v=3.0, lid=0.2, Kn=0.4, mass_rescale=0)
    mac = inputs.random_macros(p, 7)
    o = Oracle(p, mac)
    w_in = o.rho_w().copy()
    o.iterate(1)
    ref, ref_w = o.macros(), o.rho_w()
    for precision, tol in ((kgs.KGS_FP64, FP64_TOL), (kgs.KGS_MIXED, MIXED_TOL)):
        c = kgs.kgs_setup(p, precision=precision)
        kgs.kgs_set_initial(c, mac)
        assert kgs.kgs_iterate(c, 1)[0] == kgs.KGS_OK
        assert_fields_close(kgs.kgs_moments(c), ref, tol, what="context, %s" % precision)
        assert_rho_w_close(kgs.kgs_rho_w(c), ref_w, tol)
    b = kgs.kgs_batch_setup([p, p], precision=kgs.KGS_MIXED, v_per_cta=256, block_z=8)
    for i in range(2):
        kgs.kgs_batch_set_initial(b, i, mac)
    assert kgs.kgs_batch_iterate(b, 1)[0] == kgs.KGS_OK
    assert_fields_close(kgs.kgs_batch_moments(b, 1), ref, MIXED_TOL, what="batch")
    m_in, w_dev = torch.tensor(mac, device="cuda"), torch.tensor(w_in, device="cuda")
    m, w = torch.empty_like(m_in), torch.empty_like(w_dev)
    rc, _ = kgs.kgs_iterate_noalloc(p, m_in.data_ptr(), w_dev.data_ptr(), m.data_ptr(), w.data_ptr(),
                                    precision=kgs.KGS_MIXED)
    assert rc == kgs.KGS_OK
    assert_fields_close(m.cpu().numpy().reshape(mac.shape), ref, MIXED_TOL, what="no allocation")
    assert_rho_w_close(w.cpu().numpy(), ref_w, MIXED_TOL)
