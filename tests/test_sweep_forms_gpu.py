"""The separated FP64 sweep and the packed FP32 sweep over the forms that their
tables and slot orders depend on: velocity axes of one, two and few nodes, odd
counts (a node at zero), lines longer than a group's half, axes whose nodes
are not sorted, and blocks of every depth, with ragged tails and solid cells.

References: the FP64 oracle, and for FP64 also the general sweep, which serves
the entry point without device allocation.  Tolerances are those of the
parity tests: 1e-10 (FP64) and 1e-5 (mixed).
"""
import dataclasses

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


def problem(cells, vels, unsorted=False, solid=False, widths=False, **kw):
    p = inputs.cavity(cells, vels, L_v=3.0, lid=0.2, Kn=0.4, **kw)
    rng = np.random.default_rng(11)
    if unsorted:
        change = {}
        for a in "xyz":
            k = rng.permutation(len(getattr(p, "xi_" + a)))
            change["xi_" + a], change["w_" + a] = getattr(p, "xi_" + a)[k], getattr(p, "w_" + a)[k]
        p = dataclasses.replace(p, **change)
    if widths:
        p = dataclasses.replace(p, dx=p.dx * rng.uniform(0.7, 1.3, p.nx), dz=p.dz * rng.uniform(0.7, 1.3, p.nz))
    if solid:
        s = np.zeros((p.nz, p.ny, p.nx), np.uint8)
        s[3:6, 2:5, 4:9] = 1
        p = dataclasses.replace(p, solid=s)
    return p


FORMS = [
    dict(cells=[9, 10, 7], vels=[1, 3, 2]),
    dict(cells=[9, 8, 7], vels=[2, 2, 2]),
    dict(cells=[5, 9, 6], vels=[3, 4, 5]),
    dict(cells=[9, 10, 11], vels=[9, 7, 8], unsorted=True),
    dict(cells=[8, 8, 9], vels=[17, 5, 6], unsorted=True, widths=True),
    dict(cells=[17, 9, 9], vels=[11, 12, 9], solid=True),
    dict(cells=[17, 16, 10], vels=[32, 5, 6], solid=True, widths=True),
    dict(cells=[4, 9, 3], vels=[300, 2, 3]),
    dict(cells=[4, 9, 3], vels=[2, 2, 290]),
]


@pytest.mark.parametrize("form", range(len(FORMS)))
@pytest.mark.parametrize("block_z", [1, 3, 0])
def test_forms_against_oracle(kgs, form, block_z):
    p = problem(**FORMS[form])
    mac = inputs.random_macros(p, 5 + form)
    o = Oracle(p, mac)
    o.iterate(2)
    for precision, tol in ((kgs.KGS_FP64, FP64_TOL), (kgs.KGS_MIXED, MIXED_TOL)):
        c = kgs.kgs_setup(p, precision=precision, block_z=block_z)
        kgs.kgs_set_initial(c, mac)
        rc, _, _ = kgs.kgs_iterate(c, 2)
        assert rc == kgs.KGS_OK
        assert_fields_close(kgs.kgs_moments(c), o.macros(), tol, solid=p.solid, what="%s, %s" % (FORMS[form], precision))
        # a wall that no velocity crosses has no wall density (0 / 0 in the oracle)
        rw = o.rho_w()
        assert_rho_w_close(np.where(np.isnan(rw), 0.0, kgs.kgs_rho_w(c)), np.nan_to_num(rw, nan=0.0), tol)


# the general FP64 sweep's tables hold lines of up to about 100 nodes
@pytest.mark.parametrize("form", [i for i, f in enumerate(FORMS) if f["vels"][0] <= 100])
def test_separated_fp64_against_general_sweep(kgs, form):
    import torch

    p = problem(**FORMS[form], mass_rescale=0)
    mac = inputs.random_macros(p, 50 + form)
    c = kgs.kgs_setup(p, precision=kgs.KGS_FP64)
    kgs.kgs_set_initial(c, mac)
    w_in = torch.tensor(kgs.kgs_rho_w(c), device="cuda")
    m_in = torch.tensor(mac, device="cuda")
    m, w = torch.empty_like(m_in), torch.empty_like(w_in)
    rc, res = kgs.kgs_iterate_noalloc(p, m_in.data_ptr(), w_in.data_ptr(), m.data_ptr(), w.data_ptr(),
                                      precision=kgs.KGS_FP64)
    assert rc == kgs.KGS_OK
    rc, _, r = kgs.kgs_iterate(c, 1)
    assert rc == kgs.KGS_OK
    assert_fields_close(kgs.kgs_moments(c), m.cpu().numpy(), FP64_TOL, solid=p.solid, what=str(FORMS[form]))
    assert_rho_w_close(kgs.kgs_rho_w(c), w.cpu().numpy(), FP64_TOL)
    assert abs(r - res) <= 1e-8 * res
