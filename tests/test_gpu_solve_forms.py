"""Mixed solves whose filters run in the J form at the edges of its tiles (256 rows of 2n, columns
of 2 (nev + nex) around 32 and 64), and in the blocks form with its correction source (few
columns of a large matrix, and the fallback Rayleigh-Ritz), against the FP64-accurate solve."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2601_10557_gb300 as p
    if not p.has_mixed():
        pytest.fail("tensor-core filter not available on this device")
    return p


def _problem(n, low, seed):
    """A = F diag(d) F^* with `low` separated values below the rest, B a weak symmetric coupling."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    d = torch.cat([torch.linspace(1.0, 2.0, low, dtype=torch.float64),
                   torch.linspace(4.0, 9.0, n - low, dtype=torch.float64)]).cuda()
    ph = torch.polar(torch.ones_like(d), 6.2831853 * torch.rand(n, generator=g, dtype=torch.float64, device="cuda"))
    A = torch.fft.fft(torch.diag(d).to(torch.complex128), dim=0, norm="ortho") * ph[:, None]
    A = torch.fft.ifft(A, dim=1, norm="ortho") * ph.conj()[None, :]
    G = torch.randn((n, n), generator=g, dtype=torch.complex128, device="cuda")
    return ((A + A.conj().T) * 0.5).contiguous(), ((G + G.T) * (0.1 / np.sqrt(n))).contiguous()


@pytest.mark.parametrize("n,nev,nex,rr", [(63, 4, 4, "oblique"), (127, 7, 9, "oblique"), (128, 8, 8, "oblique"),
                                          (129, 9, 8, "oblique"), (257, 20, 13, "oblique"),
                                          (129, 9, 8, "fallback"), (3001, 3, 4, "oblique")])
def test_mixed_solve_matches_the_fp64_accurate_one(pkg, n, nev, nex, rr):
    A, B = _problem(n, nev + nex, n)
    tol = 1e-10
    out = {}
    for p in ("fp64_tc", "mixed"):
        lam, V, st = pkg.solve(A, B, nev, nex, 8, tol, precision=p, deg_max=20, maxiter=40, seed=3, rr=rr)
        n2 = V.shape[1] // 2
        X, Y = V[:, :n2], V[:, n2:]
        R = torch.cat([X @ A.T + Y @ B.T, -(X @ B.conj().T) - (Y @ A.conj().T)], 1) - lam[:, None] * V
        assert float(torch.linalg.vector_norm(R, dim=1).max()) <= 1.01 * tol * st["rho_hat"]
        out[p] = lam.cpu().numpy()
    # a residual of tol rho_hat moves an eigenvalue of this well-conditioned problem by less than that
    np.testing.assert_allclose(out["mixed"], out["fp64_tc"], rtol=0, atol=20 * tol)
