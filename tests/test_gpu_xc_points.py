"""The FP64 exchange-correlation potential entry by entry: its elementary
functions (cube root, inverse root, reciprocal, logarithm) over the whole range
of densities, not against the largest entry.  Without atoms' charge and Hartree
potential V_eff is v_xc alone."""
import numpy as np
import pytest

import ks_inputs as ki
from oracle import energy as oe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -53
RS1 = 3.0 / (4.0 * np.pi)                     # density of r_s = 1


def potential(rho, xc, **kw):
    import paper_1308_2864_gb300 as ks
    N = round(len(rho) ** (1 / 3))
    s = ki.small_system(N=N, L=5.0, natoms=1, p=1, Z=0.0, seed=1)
    s.xc = xc
    P = ks.Problem.from_system(s, **kw)
    zero = torch.zeros(s.n, dtype=torch.float64, device="cuda")
    veff, e = P.step_potential(torch.from_numpy(rho).cuda(), zero, None)
    return veff.cpu().numpy(), e, s


@pytest.mark.parametrize("xc", [0, 1])
@pytest.mark.parametrize("lo,hi", [(1e-30, 1e-12), (1e-12, 1e-3), (1e-3, 0.99 * RS1),
                                   (0.99 * RS1, 1.01 * RS1), (1.01 * RS1, 1e3), (1e3, 1e12)])
def test_xc_potential_per_entry(xc, lo, hi):
    # every term of v_xc has the same sign, so no digit cancels: at most 16
    # roundings here and 16 in the oracle's own double evaluation
    rho = lo * (hi / lo) ** np.random.default_rng(7).random(20 ** 3)
    rho[:2] = lo, hi
    got, e, s = potential(rho, xc)
    eps, want = oe.lda(rho, xc)
    assert np.all(np.abs(got - want) <= 32 * U * np.abs(want))
    h3 = (s.L / (s.N + 1)) ** 3
    assert e[2] == pytest.approx(h3 * float(rho @ eps), rel=1e-13)


def test_density_floor_and_joint():
    # below the floor nothing, at it the formula; r_s = 1 is continuous to the
    # parametrisation's own joint (C and D make eps_c and v_c meet)
    rho = np.full(8, 0.1)
    rho[:6] = [0.0, 9.9e-31, 1e-30, -1.0, RS1 * (1 - 4 * U), RS1 * (1 + 4 * U)]
    got, _, _ = potential(rho, 1)
    assert got[0] == got[1] == got[3] == 0.0 and got[2] < 0.0
    assert abs(got[4] - got[5]) <= 64 * U * abs(got[4])


@pytest.mark.parametrize("rho_big", [1e39, 1e300, np.inf])
def test_density_beyond_the_fp32_starts_is_not_a_number(rho_big):
    # r_s underflows there: the correlation energy is not a finite number, and a
    # call that evaluates it reports KS_ENAN instead of an energy
    rho = np.full(27, 0.3)
    rho[13] = rho_big
    _, e, _ = potential(rho, 1)
    assert not np.isfinite(e[2])
