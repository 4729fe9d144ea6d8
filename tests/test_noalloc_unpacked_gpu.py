"""Mixed problems whose tables fit the fixed scratch of kgs_iterate_noalloc only
without the packed velocity slots (short x-lines: their table of lines is as
long as the velocity grid): they run on the unpacked sweep of one launch per
stage, and agree with an FP64 context to the tolerance of the mixed path.
"""
import pytest

from paper_1810_00348_gb300 import inputs
from tests.parity import assert_fields_close, assert_rho_w_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kgs():
    from paper_1810_00348_gb300 import kgs as k
    k.load()
    return k


# bytes below the limit without, above it with the packed slots: 50432 / 52224 and 47104 / 40704
@pytest.mark.parametrize("cells,vels", [([38, 14, 32], [2, 40, 40]), ([24, 24, 33], [2, 36, 38])])
def test_fits_only_without_packed_slots(kgs, cells, vels):
    import torch

    p = inputs.cavity(cells, vels, lid=0.2, Kn=0.4, mass_rescale=0)
    mac = inputs.random_macros(p, 9)
    c = kgs.kgs_setup(p, precision=kgs.KGS_FP64)
    kgs.kgs_set_initial(c, mac)
    w_in, m_in = torch.tensor(kgs.kgs_rho_w(c), device="cuda"), torch.tensor(mac, device="cuda")
    m, w = torch.empty_like(m_in), torch.empty_like(w_in)
    rc, _ = kgs.kgs_iterate_noalloc(p, m_in.data_ptr(), w_in.data_ptr(), m.data_ptr(), w.data_ptr(),
                                    precision=kgs.KGS_MIXED)
    assert rc == kgs.KGS_OK
    assert kgs.kgs_iterate(c, 1)[0] == kgs.KGS_OK
    assert_fields_close(m.cpu().numpy(), kgs.kgs_moments(c), 1e-5, what="unpacked")
    assert_rho_w_close(w.cpu().numpy(), kgs.kgs_rho_w(c), 1e-5)
    bigger = inputs.cavity([n + 2 for n in cells], vels, lid=0.2, Kn=0.4, mass_rescale=0)
    with pytest.raises(kgs.KgsError):
        kgs.kgs_iterate_noalloc(bigger, m_in.data_ptr(), w_in.data_ptr(), m.data_ptr(), w.data_ptr(),
                                precision=kgs.KGS_MIXED)
