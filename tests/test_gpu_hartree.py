"""The Hartree solver's sine transforms in parity form against the exact sine
solve, at the edges of their tiles: the smallest grids, odd and even edges (a
middle node or none), 64 / 65 (2 x 2 to 4 x 4 outputs per thread), 128 / 129
(in-plane to tiled axis passes).  Same tolerances as the general Hartree test:
the oracle's residual within 5 % of cg_tol, the potential at 1e-8."""
import math

import numpy as np
import pytest

import ks_inputs as ki
from oracle import fe as ofe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [2, 3, 4, 7, 8, 9, 17, 24, 31, 63, 64, 65, 81, 127, 128, 129])
def test_hartree_parity_transforms(N):
    import paper_1308_2864_gb300 as ks
    s = ki.small_system(N=N, L=0.4 * (N + 1), natoms=1, p=1, Z=2.0, seed=N)
    P = ks.Problem.from_system(s)
    rho = np.random.default_rng(N).random(N ** 3) + 0.1
    b = 4 * math.pi * s.h ** 3 * rho
    exact = ofe.poisson_exact(b, N, s.h)
    v, _, it = P.step_hartree(torch.from_numpy(rho).cuda())
    v = v.cpu().numpy()
    res = b - ofe.apply_K(v, N, s.h)
    assert np.linalg.norm(res) <= 1.05e-10 * np.linalg.norm(b)
    assert np.abs(v - exact).max() <= 1e-8 * np.abs(exact).max()
    assert it <= 4
    # a warm start from a different potential reaches the same one
    w = torch.from_numpy(0.9 * exact + 0.01 * rho).cuda()
    w, _, _ = P.step_hartree(torch.from_numpy(rho).cuda(), w, warm=True)
    assert np.abs(w.cpu().numpy() - exact).max() <= 1e-8 * np.abs(exact).max()
