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


@pytest.mark.parametrize("graphs", [True, False])
def test_stalled_correction_goes_on_as_conjugate_gradients(graphs):
    # at a node spacing of 3e19 the products of two 1-D eigenvalues overflow FP32
    # for half of the modes: the sine-basis inverse leaves them out, the
    # correction stalls, and both paths finish with CG.  A job table holds such a
    # job beside an ordinary one.  Energies at the Hartree tolerance (1e-10 of the
    # residual): 1e-8, as the potential above.
    import paper_1308_2864_gb300 as ks
    from oracle import energy as oe
    wide = ki.small_system(N=9, L=3e20, natoms=1, p=1, Z=2.0, seed=3)
    usual = ki.small_system(N=10, L=7.0, natoms=2, p=2, Z=1.0, seed=7)
    P = ks.Problem.from_system(wide)
    # (x0() is bound to the atom; norms near 1, as the factor's FP32 starts need)
    x0 = np.random.default_rng(5).standard_normal((wide.n, 1)) / math.sqrt(wide.n * wide.h ** 3)
    X = torch.from_numpy(x0).cuda()
    P.orthonormalize(X)
    rho = P.step_density(X)
    _, _, it = P.step_hartree(rho)
    assert 4 < it < 200
    E = P.energy_grad(X)[0]
    assert E == pytest.approx(oe.evaluate(oe.Model.from_system(wide), X.cpu().numpy()).E, rel=1e-8)
    B = ks.Batch([usual, wide])
    B.set_graphs(graphs)
    res, _ = B.minimize([usual.x0(), x0], gtol=1e30, maxit=1)
    assert [r["status"] for r in res] == [0, 0]
    assert res[1]["E"] == pytest.approx(E, rel=1e-8)
    assert res[1]["cg_iters_total"] < 200
