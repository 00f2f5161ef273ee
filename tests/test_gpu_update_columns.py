"""The pipelined FP32 update of up to 64 columns at its column counts: the
epilogue's operand (Bm, or the base X_b of the increment form) comes through
the ring in stages of 32 columns, one where the row has no more, two above.
In the bounds-checked build a stage past the row's end is on record."""
import numpy as np
import pytest

import ks_inputs as ki
from oracle import energy as oe
from oracle import stiefel as ost

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k1,k2,q", [(96, 0, 32), (96, 96, 32), (96, 64, 20), (72, 0, 4),
                                     (68, 36, 36), (96, 0, 64), (64, 64, 64), (32, 32, 64)])
def test_update_columns(k1, k2, q):
    # above 64 values of K the pipelined kernel also serves q <= 32.  Each output
    # is one chain of k1 + k2 FMAs and two more roundings, of operands rounded once.
    import paper_1308_2864_gb300 as ks
    for N in (5, 13):
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


@pytest.mark.parametrize("retraction", ["qr", "cayley"])
def test_increment_form_of_32_orbitals(retraction):
    # K = 96, q = 32: the retraction with X_b as the second output's operand.  The
    # tolerance is that of the wide increment test: 1e-6 of the energy's terms.
    import paper_1308_2864_gb300 as ks
    s = ki.small_system(N=14, L=8.0, natoms=4, p=32, Z=4.0, seed=11)
    model = oe.Model.from_system(s)
    P = ks.Problem.from_system(s)
    X = torch.from_numpy(np.ascontiguousarray(s.x0())).cuda()
    r = P.minimize(X, retraction=retraction, gtol=1e-12, maxit=12, precision="mixed",
                   stall_iters=0)
    assert r["mixed_iters"] == 12 and r["status"] == ks.KS_ENOCONV
    ev = oe.evaluate(model, X.cpu().numpy())
    scale = sum(abs(v) for v in ev.parts.values())
    assert abs(r["E"] - ev.E) <= 1e-6 * scale
    assert ost.ortho_error(model, X.cpu().numpy()) < 1e-6


@pytest.mark.parametrize("q", [12, 15, 16, 17, 26, 32])
def test_narrow_update_forms(q):
    # 48^3 rows fill the chip: staged tiles from 16 columns on, one row per thread
    # below; at 12^3 one row per thread up to K = 32.  Both are one chain over k.
    import paper_1308_2864_gb300 as ks
    for N, blocks in ((12, 1), (12, 2), (48, 1), (48, 2)):
        s = ki.small_system(N=N, L=7.0, natoms=2, p=q, Z=4.0, seed=4)
        P = ks.Problem.from_system(s)
        g = torch.Generator(device="cuda").manual_seed(q)
        r = lambda *d: torch.randn(*d, generator=g, device="cuda", dtype=torch.float64)
        A, Bm = [r(s.n, q).float() for _ in range(blocks)], r(s.n, q).float()
        C = [r(q, q) for _ in range(blocks)]
        two = (A[1], C[1]) if blocks == 2 else (None, None)
        torch.cuda.synchronize()             # the problem has a stream of its own
        got = P.step_combine_f32(A[0], C[0], *two, alpha=-0.5, beta=2.0, Bm=Bm).double()
        want, bound = 2.0 * Bm.double(), 2.0 * Bm.double().abs()
        for a, c in zip(A, C):
            want = want - 0.5 * (a.double() @ c)
            bound = bound + 0.5 * (a.double().abs() @ c.abs())
        assert torch.all((got - want).abs() <= (blocks * q + 4) * 2.0**-23 * bound)


@pytest.mark.parametrize("N,k1,k2,q", [(28, 36, 36, 36), (28, 72, 4, 257), (29, 256, 256, 256),
                                       (28, 300, 260, 300), (24, 256, 256, 256),
                                       (10, 640, 640, 640), (9, 644, 640, 300)])
def test_wide_update_tiles(N, k1, k2, q):
    # 256-row tiles: grids of more than one wave of 128-row tiles, or K above 1024;
    # 128-row tiles otherwise (24^3 x 256).  The bound of the general tensor-core test
    import paper_1308_2864_gb300 as ks
    s = ki.small_system(N=N, L=7.0, natoms=2, p=max(k1, k2, q), Z=4.0, seed=4)
    P = ks.Problem.from_system(s)
    P.set_tensor_cores(2)
    g = torch.Generator(device="cuda").manual_seed(29)
    r = lambda *d: torch.randn(*d, generator=g, device="cuda", dtype=torch.float64)
    A1, A2, Bm, C1, C2 = (r(s.n, k1).float(), r(s.n, k2).float(), r(s.n, q).float(), r(k1, q),
                          r(k2, q))
    torch.cuda.synchronize()                 # the problem has a stream of its own
    for bm, beta in ((None, 0.0), (Bm, 2.0)):
        got = P.step_combine_f32(A1, C1, A2, C2, alpha=-0.5, beta=beta, Bm=bm).double()
        want = -0.5 * (A1.double() @ C1 + A2.double() @ C2) + beta * Bm.double()
        bound = (0.5 * (A1.double().abs() @ C1.abs() + A2.double().abs() @ C2.abs())
                 + beta * Bm.double().abs())
        assert torch.all((got - want).abs() <= 4e-6 * bound + 1e-12)
