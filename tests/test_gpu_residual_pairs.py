"""Residual norms of converged pairs: differences at the rounding level of their terms.  H is
diagonally dominant (the usual Bethe-Salpeter case) or graded, so that the largest entries of a row
and of a vector say little about the products that occur in a sum."""
import numpy as np
import pytest
import torch

from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2601_10557_gb300 as p
    p.lib()
    return p


def _problem(kind, n):
    rng = np.random.default_rng(n)
    d = np.linspace(1.0, 10.0, n) if kind == "dominant" else np.logspace(0.0, 7.0, n)
    G = rng.standard_normal((2, n, n)) + 1j * rng.standard_normal((2, n, n))
    A = np.diag(d) + 0.0125 / np.sqrt(n) * (G[0] + G[0].conj().T)
    return A, 0.0125 / np.sqrt(n) * (G[1] + G[1].T)


def _pairs(A, B, k):
    """k eigenpairs by correcting each row of (H - lambda) v = 0 by its diagonal, from unit vectors."""
    n = A.shape[0]
    H = np.block([[A, B], [-B.conj(), -A.conj()]])
    V, lam = np.zeros((k, 2 * n), complex), np.zeros(k)
    for j in range(k):
        m = j * (n // k)
        z = np.zeros(2 * n, complex)
        z[m] = 1.0
        for _ in range(60):
            t = H @ z
            r = t - t[m].real * z
            r[m] = 0.0
            D = np.diag(H) - t[m].real
            D[m] = 1.0
            z = z - r / D
        lam[j] = (H @ z)[m].real
        V[j] = z / np.linalg.norm(z)
    return V, lam


@pytest.mark.parametrize("kind", ["dominant", "graded"])
@pytest.mark.parametrize("n,k", [(96, 6), (512, 32)])
def test_residuals_of_converged_pairs(pkg, kind, n, k):
    A, B = _problem(kind, n)
    V, lam = _pairs(A, B, k)
    got = pkg.residuals(to_dev(A), to_dev(B), to_dev(V), torch.from_numpy(lam).cuda()).cpu().numpy()
    wide = [M.astype(np.clongdouble) for M in (A, B, V[:, :n], V[:, n:])]
    Al, Bl, X, Y = wide
    l = lam.astype(np.longdouble)[:, None]
    R = np.concatenate([X @ Al.T + Y @ Bl.T - l * X, -(X @ Bl.conj().T) - (Y @ Al.conj().T) - l * Y], 1)
    ref = np.sqrt((np.abs(R) ** 2).sum(1)).astype(float)
    # an FP64 sum of 2n complex products is off by up to 4n 2^-53, and mostly by sqrt(4n) 2^-53, of
    # the sum of its terms' magnitudes (lambda w among them)
    S = np.concatenate([np.abs(X) @ np.abs(Al).T + np.abs(Y) @ np.abs(Bl).T + np.abs(l * X),
                        np.abs(X) @ np.abs(Bl).T + np.abs(Y) @ np.abs(Al).T + np.abs(l * Y)], 1)
    terms = np.sqrt((S ** 2).sum(1)).astype(float)
    assert (np.abs(got - ref) <= np.sqrt(4.0 * n) * 2.0 ** -53 * terms).all()
