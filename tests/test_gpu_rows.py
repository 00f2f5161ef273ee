"""The FP64 row kernels (symmetric Gram, triangular update, row update) through
the calls that use them, against the oracle, at the edges of their blocks:
9 and 128 are the ends of the range, 36 and 37 leave whole and ragged blocks of
four columns, 33 and 127 have an odd row pitch; the grids leave ragged row
tiles and fewer tiles than SMs.  Tolerance: the parity tests' 1e-12 relative
for one product, 1e-11 for the products chained behind a Cholesky factor."""
import numpy as np
import pytest

import ks_inputs as ki
from oracle import energy as oe
from oracle import stiefel as ost

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def assert_rel(got, want, rel, what):
    got, want = np.asarray(got), np.asarray(want)
    err = np.abs(got - want).max() / max(np.abs(want).max(), 1e-300)
    assert err <= rel, f"{what}: {err:.3e} > {rel:.1e}"


@pytest.mark.parametrize("N,p", [(7, 9), (11, 33), (13, 36), (13, 37), (11, 64), (9, 127),
                                 (11, 128), (9, 130)])
def test_row_kernels(N, p):
    import paper_1308_2864_gb300 as ks
    s = ki.small_system(N=N, L=6.0, natoms=2, p=p, Z=4.0, seed=21 + p)
    model = oe.Model.from_system(s)
    P = ks.Problem.from_system(s, cg_tol=1e-13)
    X0 = s.x0()
    X = ost.m_orthonormalize(model, X0)
    Xd = dev(X0)
    P.orthonormalize(Xd)
    Xh = Xd.cpu().numpy()
    assert_rel(Xh, X, 1e-11, "orthonormalize")
    assert np.linalg.norm(Xh.T @ model.apply_M(Xh) - np.eye(p)) <= 1e-12 * np.sqrt(p)
    pt = ost.point_at(model, X)
    E, EX, D, g = P.energy_grad(dev(X), want_ex=True, want_d=True)
    assert abs(E - pt.ev.E) <= 1e-11 * abs(pt.ev.E)
    assert_rel(EX.cpu().numpy(), pt.ev.EX, 1e-10, "E_X")
    assert_rel(D.cpu().numpy(), pt.D, 1e-9, "D")
    assert abs(g - pt.dnorm) <= 1e-9 * pt.dnorm
    # an energy alone (no gradient stored) is the same energy
    assert P.energy_grad(dev(X), want_ex=False)[0] == pytest.approx(E, rel=1e-12)
    for kind, ref in ((ks.KS_QR, ost.retract_qr), (ks.KS_CAYLEY, ost.retract_cayley)):
        got = P.retract(kind, dev(X), dev(pt.ev.EX), 0.01).cpu().numpy()
        assert_rel(got, ref(model, pt, 0.01), 1e-11, f"retract {kind}")


def test_retract_takes_any_derivative_block():
    # E_X of a caller need not come from a symmetric H: E_X^T X is then not symmetric
    import paper_1308_2864_gb300 as ks
    s = ki.small_system(N=11, L=6.0, natoms=2, p=20, Z=4.0, seed=5)
    model = oe.Model.from_system(s)
    X = ost.m_orthonormalize(model, s.x0())
    ev = oe.evaluate(model, X)
    ev.EX = np.random.default_rng(3).standard_normal(X.shape)
    pt = ost.project(model, X, ev)
    P = ks.Problem.from_system(s)
    got = P.retract(ks.KS_CAYLEY, dev(X), dev(ev.EX), 1e-3).cpu().numpy()
    assert_rel(got, ost.retract_cayley(model, pt, 1e-3), 1e-11, "retract")
    bad = ev.EX.copy()
    bad[17, 3] = np.nan
    for kind in (ks.KS_QR, ks.KS_CAYLEY):
        with pytest.raises(ks.KSError) as e:
            P.retract(kind, dev(X), dev(bad), 1e-3)
        assert e.value.status == ks.KS_ENAN


@pytest.mark.parametrize("p", [2, 3, 4, 17, 68, 69])
def test_cayley_factor_sizes(p):
    # 68 | 69: the 2p x 3p system in shared memory | in global scratch; a large step, so
    # that rows are exchanged.  1e-11: as the other retractions above
    import paper_1308_2864_gb300 as ks
    s = ki.small_system(N=9, L=5.0, natoms=2, p=p, Z=4.0, seed=60 + p)
    model = oe.Model.from_system(s)
    X = ost.m_orthonormalize(model, s.x0())
    pt = ost.point_at(model, X)
    P = ks.Problem.from_system(s, cg_tol=1e-13)
    for tau in (1e-3, 0.5):
        got = P.retract(ks.KS_CAYLEY, dev(X), dev(pt.ev.EX), tau).cpu().numpy()
        assert_rel(got, ost.retract_cayley(model, pt, tau), 1e-11, f"tau {tau}")


@pytest.mark.parametrize("N,k1,k2,q", [(4, 36, 36, 33), (7, 40, 36, 260), (7, 256, 256, 256),
                                       (8, 300, 260, 300), (10, 260, 4, 257), (12, 512, 512, 512)])
def test_wide_fp32_update_on_tensor_cores(N, k1, k2, q):
    # widths that are multiples of 4 (the pipelined form): K of 72 .. 1024 in
    # stages of 16 with a ragged last one, fewer rows than a tile (4^3) and ragged
    # row and column tiles; the bound of the general tensor-core update test
    import paper_1308_2864_gb300 as ks
    s = ki.small_system(N=N, L=7.0, natoms=2, p=max(k1, k2, q), Z=4.0, seed=4)
    P = ks.Problem.from_system(s)
    P.set_tensor_cores(2)
    rng = np.random.default_rng(29)
    A1 = rng.standard_normal((s.n, k1)).astype(np.float32)
    A2 = rng.standard_normal((s.n, k2)).astype(np.float32)
    Bm = rng.standard_normal((s.n, q)).astype(np.float32)
    C1, C2 = rng.standard_normal((k1, q)), rng.standard_normal((k2, q))
    t = lambda a: torch.from_numpy(a).cuda()
    A1d, A2d = A1.astype(np.float64), A2.astype(np.float64)
    for bm, beta in ((None, 0.0), (Bm, 2.0)):
        got = P.step_combine_f32(t(A1), t(C1), t(A2), t(C2), alpha=-0.5, beta=beta,
                                 Bm=None if bm is None else t(bm)).cpu().numpy()
        want = -0.5 * (A1d @ C1 + A2d @ C2) + beta * Bm
        bound = 0.5 * (np.abs(A1d) @ np.abs(C1) + np.abs(A2d) @ np.abs(C2)) + beta * np.abs(Bm)
        assert np.all(np.abs(got - want) <= 4e-6 * bound + 1e-12)


@pytest.mark.parametrize("pa,qb", [(9, 9), (16, 16), (16, 17), (17, 16), (9, 29), (31, 31),
                                   (32, 31), (31, 32), (32, 32)])
def test_mid_gram_thread_blocks(pa, qb):
    # both sides of 256 outputs (one or 2 x 2 per thread), odd widths; rows that
    # end inside a stage of 32.  A chain of n rounded products: n unit roundoffs.
    import paper_1308_2864_gb300 as ks
    for N in (4, 9):
        s = ki.small_system(N=N, L=7.0, natoms=2, p=max(pa, qb), Z=4.0, seed=4)
        P = ks.Problem.from_system(s)
        rng = np.random.default_rng(pa * 40 + qb)
        A, B = rng.standard_normal((s.n, pa)), rng.standard_normal((s.n, qb))
        got = P.step_gram(dev(A), dev(B)).cpu().numpy()
        assert np.all(np.abs(got - A.T @ B) <= 2 * s.n * 2.0**-53 * (np.abs(A).T @ np.abs(B)))
        A, B = A.astype(np.float32), B.astype(np.float32)
        got = P.step_gram_f32(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()).cpu().numpy()
        A, B = A.astype(np.float64), B.astype(np.float64)
        assert np.all(np.abs(got - A.T @ B) <= 2 * s.n * 2.0**-24 * (np.abs(A).T @ np.abs(B)))


@pytest.mark.parametrize("k1,k2,q", [(1, 0, 1), (4, 4, 4), (5, 5, 5), (8, 8, 8), (17, 17, 17),
                                     (26, 26, 26), (31, 30, 29), (32, 32, 32), (33, 64, 3),
                                     (64, 63, 32)])
def test_narrow_fp32_update_tiles(k1, k2, q):
    # column groups with and without a remainder, K in one stage, two and a stage
    # of one; rows that end inside a tile.  Each output is one chain of k1 + k2 FMAs
    # and two more roundings, of operands rounded once.
    import paper_1308_2864_gb300 as ks
    for N in (4, 12):
        s = ki.small_system(N=N, L=7.0, natoms=2, p=max(k1, k2, q), Z=4.0, seed=4)
        P = ks.Problem.from_system(s)
        rng = np.random.default_rng(k1 + 100 * q)
        t = lambda a: torch.from_numpy(a).cuda()
        f32 = lambda k: rng.standard_normal((s.n, k)).astype(np.float32)
        A1, A2, Bm = f32(k1), f32(k2), f32(q)
        C1, C2 = rng.standard_normal((k1, q)), rng.standard_normal((k2, q))
        for bm, beta in ((None, 0.0), (Bm, 2.0)):
            two = (t(A2), t(C2)) if k2 else (None, None)
            got = P.step_combine_f32(t(A1), t(C1), *two, alpha=-0.5, beta=beta,
                                     Bm=None if bm is None else t(bm)).cpu().numpy()
            want = -0.5 * (A1.astype(float) @ C1 + A2.astype(float) @ C2) + beta * Bm
            bound = 0.5 * (np.abs(A1).astype(float) @ np.abs(C1)
                           + np.abs(A2).astype(float) @ np.abs(C2)) + beta * np.abs(Bm)
            assert np.all(np.abs(got - want) <= (k1 + k2 + 4) * 2.0**-23 * bound)
