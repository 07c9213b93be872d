"""Statuses of solves on indefinite S H: the non-hermitian fallback runs in every iteration, and
a solve that reaches maxiter returns its statistics with NOT_CONVERGED like any other."""
import numpy as np
import pytest
import torch

import bse_inputs as bi
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2601_10557_gb300 as p
    p.lib()
    return p


def _indefinite(n, nneg, diagonal):
    """A with nneg negative eigenvalues, weakly coupled: H has real eigenvalues, S H is indefinite."""
    rng = np.random.default_rng(n + nneg)
    d = np.linspace(2.0, 6.0, n)
    d[:nneg] = -np.linspace(1.0, 1.3, nneg)
    G = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    U = np.eye(n) if diagonal else bi.haar_unitary(n, rng)
    A = ((U * d) @ U.conj().T).astype(complex)
    return to_dev((A + A.conj().T) / 2), to_dev(0.02 / np.sqrt(n) * (G + G.T))


@pytest.mark.parametrize("precision", ["fp64", "mixed", "fp64_tc"])
@pytest.mark.parametrize("nneg,diagonal", [(1, False), (2, True), (4, False)])
def test_indefinite_solve_at_maxiter_is_not_converged(pkg, precision, nneg, diagonal):
    A, B = _indefinite(32, nneg, diagonal)
    lam, V, st = pkg.solve(A, B, 4, 4, 8, 1e-10, precision=precision, maxiter=1, allow_partial=True)
    assert st["status"] == 1 and st["iterations"] == 1 and st["converged"] < 4
    # one negative direction can lie outside the first search space
    assert st["fallback_rr"] == 1 or nneg == 1


def test_indefinite_solve_converges_by_the_fallback(pkg):
    A, B = _indefinite(32, 2, False)
    lam, V, st = pkg.solve(A, B, 4, 4, 8, 1e-10)
    H = torch.cat([torch.cat([A, B], 1), torch.cat([-B.conj(), -A.conj()], 1)])
    R = V @ H.T - lam[:, None] * V
    assert st["fallback_rr"] > 0 and float(torch.linalg.vector_norm(R, dim=1).max()) <= 1e-9 * float(st["rho_hat"])
