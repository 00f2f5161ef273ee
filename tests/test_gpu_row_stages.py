"""The FP64 row kernels (symmetric Gram, triangular update) on enough rows for
what the small grids leave out: several stages per block of the Gram with a ragged
last one, two and four rows per thread of the update (29^3 and 45^3 rows), whole
and ragged column blocks, odd row pitches (8-byte copies).  Against plain FP64
products of torch.  Tolerances as for the small grids: 1e-12 sqrt(p) for
M-orthonormality, 1e-11 relative for products behind a Cholesky factor."""
import math

import pytest

import ks_inputs as ki

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [(29, 9), (29, 33), (29, 37), (29, 127), (29, 128), (45, 9), (45, 33), (45, 36),
         (45, 127), (45, 128)]


def rel(got, want):
    return float((got - want).abs().max() / want.abs().max())


@pytest.mark.parametrize("N,p", SIZES)
def test_orthonormalize_in_place(N, p):
    import paper_1308_2864_gb300 as ks
    s = ki.small_system(N=N, L=0.4 * (N + 1), natoms=2, p=p, Z=4.0, seed=p)
    P = ks.Problem.from_system(s)
    g = torch.Generator(device="cuda").manual_seed(N + p)
    X0 = torch.randn(s.n, p, generator=g, device="cuda", dtype=torch.float64)
    X = X0.clone()
    torch.cuda.synchronize()                 # the problem has a stream of its own
    P.orthonormalize(X)
    MX = P.step_mass(X)
    eye = torch.eye(p, device="cuda", dtype=torch.float64)
    assert float((X.T @ MX - eye).norm()) <= 1e-12 * math.sqrt(p)
    # X R = X0 with R = X^T M X0 upper triangular, positive on the diagonal
    R = MX.T @ X0
    assert rel(X @ R, X0) <= 1e-11
    assert float(torch.tril(R, -1).abs().max()) <= 1e-11 * float(R.abs().max())
    assert float(torch.diagonal(R).min()) > 0.0


@pytest.mark.parametrize("N,p", SIZES)
def test_projection_and_qr_step(N, p):
    import paper_1308_2864_gb300 as ks
    s = ki.small_system(N=N, L=0.4 * (N + 1), natoms=2, p=p, Z=4.0, seed=p)
    P = ks.Problem.from_system(s)
    g = torch.Generator(device="cuda").manual_seed(N + p)
    X = torch.randn(s.n, p, generator=g, device="cuda", dtype=torch.float64)
    torch.cuda.synchronize()
    P.orthonormalize(X)
    _, EX, D, dnorm = P.energy_grad(X, want_ex=True, want_d=True)
    want = P.step_mass_inverse(EX) - X @ (EX.T @ X)
    assert rel(D, want) <= 1e-11
    MD = P.step_mass(D)
    assert abs(dnorm - math.sqrt(float((D * MD).sum()))) <= 1e-11 * dnorm
    # the QR step: (X - tau D) L^-T with L L^T = I + tau^2 D^T M D
    tau = 0.3 / dnorm
    got = P.retract(ks.KS_QR, X, EX, tau)
    W = X - tau * D
    torch.cuda.synchronize()
    L = torch.linalg.cholesky(W.T @ P.step_mass(W))
    assert rel(got, torch.linalg.solve_triangular(L, W.T.contiguous(), upper=False).T) <= 1e-11
