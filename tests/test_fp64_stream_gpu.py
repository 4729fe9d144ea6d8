"""The FP64 moment sums keep their digits in a fast stream, where |U| is large
against the thermal speed: heat flux and temperature after one iteration
against the same iteration in numpy with sums about each cell's own velocity,
added pairwise (the oracle adds thousands of velocities one after the other,
which is less exact than what is compared here).

Tolerance.  A heat flux from sums about U^n is off by at most
gamma_m sum w f |c|^3 / 2 with m the longest chain of additions (nodes of a
line, lines of a half, groups per accumulator, accumulators, closure: below
60); for gas near a Maxwellian sum w f |c|^3 = 2.26 rho (2 R T)^(3/2).  Both
sides are allowed that much.  Sums about 0 scale with |U|^3 instead of
(2 R T)^(3/2) and with the cancelling terms of the shift: 30 times more at
Mach 5.  Fields that vary little over a block and fields that vary by a good
part of the thermal speed (amp) take the two forms of the moment phase.
"""
import dataclasses

import numpy as np
import pytest

from oracle import Oracle
from paper_1810_00348_gb300 import inputs
from tests import brute
from tests.parity import assert_fields_close, assert_rho_w_close
from tests.test_sweep_forms_gpu import FORMS, problem

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def kgs():
    from paper_1810_00348_gb300 import kgs as k
    k.load()
    return k


def iterate(p, mac, rho_w, mu_ref):
    """One outer iteration (Eqs. (2), (5), (7)): rho, T and q, [5][nz][ny][nx]."""
    xi, w = brute.velocities(p)
    m, n = mac.reshape(8, -1), p.ncell
    fluid = np.ones(n, bool) if p.solid is None else p.solid.reshape(-1) == 0
    stream, wall = brute.maxwellian(p.rho_in, p.U_in, p.T_in, xi), brute.maxwellian(1.0, np.zeros(3), p.T_solid, xi)
    width = [p.dx, p.dy, p.dz]
    f = np.zeros((n, len(w)))
    for o in range(8):
        up = [(o >> d) & 1 for d in range(3)]  # marching towards + along d
        sel = np.all((xi >= 0.0) == np.array(up, bool), axis=1)
        x, fo = xi[sel], np.zeros((n, int(sel.sum())))
        order = [range(k) if u else range(k - 1, -1, -1) for k, u in zip((p.nx, p.ny, p.nz), up)]
        for k in order[2]:
            for j in order[1]:
                for i in order[0]:
                    c = brute.cell_index(p, i, j, k)
                    if not fluid[c]:
                        continue
                    rho, U, T, q = m[0, c], m[1:4, c], m[4, c], m[5:8, c]
                    RT, v = brute.R * T, x - U
                    v2 = np.sum(v * v, axis=1)
                    fs = brute.maxwellian(rho, U, T, x)
                    fs = fs * (1.0 + (1.0 - p.Pr) * (v @ q) / (5.0 * rho * RT * RT) * (v2 / RT - 5.0))
                    rtau = rho * RT / (mu_ref * T ** p.omega)
                    num, den = rtau * fs, rtau
                    for d, at in enumerate((i, j, k)):
                        side = 2 * d + (0 if up[d] else 1)
                        nb = brute.neighbour(p, c, side)
                        g = fo[nb] if nb >= 0 else stream[sel] if nb == -1 else rho_w[side, c] * wall[sel]
                        a = np.abs(x[:, d]) / width[d][at]
                        num, den = num + a * g, den + a
                    fo[c] = num / den
        f[:, sel] = fo
    out = np.zeros((5, n))
    for c in np.flatnonzero(fluid):
        g, v = w * f[c], xi - m[1:4, c]
        rho = np.sum(g)
        v = v - np.array([np.sum(g * v[:, d]) for d in range(3)]) / rho
        v2 = np.sum(v * v, axis=1)
        out[0, c], out[1, c] = rho, np.sum(g * v2) / (3.0 * rho * brute.R)
        for d in range(3):
            out[2 + d, c] = 0.5 * np.sum(g * v2 * v[:, d])
    return out.reshape(5, p.nz, p.ny, p.nx)


@pytest.mark.parametrize("body", [False, True])
@pytest.mark.parametrize("amp", [0.05, 0.3])
@pytest.mark.parametrize("mach", [0.0, 2.0, 5.0])
def test_heat_flux_of_a_stream(kgs, mach, amp, body):
    p = inputs.cube(nx=17, ny=10, nz=9, n_vel=22, L_v=5.5, h=1.0 / 8.0, cube_lo=(0.5, 0.25, 0.25), stretched=False,
                    Kn=0.3, mach=mach, side=0.5)
    p = dataclasses.replace(p, xi_x=p.xi_x + p.U_in[0], solid=p.solid if body else None)
    mac = inputs.random_macros(p, 3, amp)
    mac[1] += p.U_in[0] * (1 if p.solid is None else p.solid == 0)
    c = kgs.kgs_setup(p, precision=kgs.KGS_FP64)
    kgs.kgs_set_initial(c, mac)
    ref = iterate(p, mac, kgs.kgs_rho_w(c).reshape(6, -1), Oracle(p).mu_ref())
    assert kgs.kgs_iterate(c, 1)[0] == kgs.KGS_OK
    got = kgs.kgs_moments(c)
    bound = 2.0 * 60.0 * EPS * 0.5 * 2.26 * np.max(ref[0] * ref[1] ** 1.5)
    err = np.max(np.abs(got[5:8] - ref[2:5]))
    assert err <= bound, "heat flux off by %g, at most %g expected" % (err, bound)
    # T = 2/3 of the second moments per mass: the same chain
    errT = np.max(np.abs(got[4] - ref[1]))
    assert errT <= 2.0 * 60.0 * EPS * np.max(ref[1])


# the sums about one velocity per slice (fields that vary little) and about
# each cell's own (fields that vary much), over the axes, grids and masks that
# the tables depend on; the tolerance is that of the FP64 parity tests
@pytest.mark.parametrize("form", range(len(FORMS)))
@pytest.mark.parametrize("amp", [0.01, 0.2])
def test_both_sums_over_forms(kgs, form, amp):
    p = problem(**FORMS[form])
    mac = inputs.random_macros(p, 30 + form, amp)
    o = Oracle(p, mac)
    c = kgs.kgs_setup(p, precision=kgs.KGS_FP64, block_z=4)
    kgs.kgs_set_initial(c, mac)
    o.iterate(1)
    assert kgs.kgs_iterate(c, 1)[0] == kgs.KGS_OK
    assert_fields_close(kgs.kgs_moments(c), o.macros(), 1e-10, solid=p.solid, what=str(FORMS[form]))
    # a wall that no velocity crosses has no wall density (0 / 0 in the oracle)
    rw = o.rho_w()
    assert_rho_w_close(np.where(np.isnan(rw), 0.0, kgs.kgs_rho_w(c)), np.nan_to_num(rw, nan=0.0), 1e-10)
