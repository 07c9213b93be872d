"""The persistent sliced GEMM at the edges of its tiles (128 x 32), chunks (128 K) and K splits,
its integer rounding to FP64, and the residual check that uses it above the FP64 pipe's break-even."""
import numpy as np
import pytest
import torch

import bse_inputs as bi
from tests.gpu_util import problem_on_device, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2601_10557_gb300 as p
    if not p.has_mixed():
        pytest.fail("tensor cores (sm_103a) not available on this device")
    return p


def _gemm(pkg, A, B, **kw):
    return pkg.dgemm_sliced(to_dev(A), to_dev(B), **kw).cpu().numpy()


# 24-bit integers: their products are held exactly, and the result is one rounding of an
# integer sum that Python forms exactly.  One split and several tiles per CTA (4096 x 1300),
# several splits (128 x 32), ragged tails of rows, columns and K.
@pytest.mark.parametrize("M,N,K", [(127, 31, 126), (128, 32, 128), (129, 33, 130), (4096, 1300, 32), (257, 65, 4096)])
def test_exact_sums_are_rounded_once(pkg, M, N, K):
    rng = np.random.default_rng(M + N + K)
    a = rng.integers(2 ** 23, 2 ** 24, size=(M, K))
    b = rng.integers(2 ** 23, 2 ** 24, size=(N, K)) * np.where(rng.random((N, 1)) < 0.5, -1, 1)
    C = _gemm(pkg, a.astype(np.float64), b.astype(np.float64))
    for r, c in zip(rng.integers(0, M, 50), rng.integers(0, N, 50)):
        exact = sum(int(x) * int(y) for x, y in zip(a[r], b[c]))  # up to 2^60: above 2^53
        assert C[r, c] == float(exact), (r, c)


@pytest.mark.parametrize("ea,eb", [(-600, -470), (-540, -530), (500, 500), (520, 480), (-400, 300)])
def test_rounding_at_the_ends_of_the_exponent_range(pkg, ea, eb):
    rng = np.random.default_rng(abs(ea))
    a = rng.integers(-2 ** 20, 2 ** 20, size=(5, 16)).astype(np.float64)
    b = rng.integers(-2 ** 20, 2 ** 20, size=(7, 16)).astype(np.float64)
    with np.errstate(over="ignore"):
        ref = np.ldexp(a @ b.T, ea + eb)  # the integer products are exact, ldexp rounds once
    assert np.array_equal(_gemm(pkg, np.ldexp(a, ea), np.ldexp(b, eb)), ref)


def test_nonfinite_rows_give_nan(pkg):
    rng = np.random.default_rng(5)
    A, B = rng.standard_normal((40, 64)), rng.standard_normal((40, 64))
    A[3, 5], B[7, 60] = np.inf, np.nan
    C = _gemm(pkg, A, B)
    bad = np.zeros((40, 40), bool)
    bad[3], bad[:, 7] = True, True
    assert np.array_equal(np.isnan(C), bad)


# below (512, 18), (1001, 9) and above the rule, odd sizes; the tolerance of the FP64 kernel's test (2n products a
# sum, errors of a few 2^-53 |H| |w| each)
@pytest.mark.parametrize("n,k", [(512, 18), (512, 77), (1001, 9), (1001, 21)])
def test_residuals_on_both_sides_of_the_rule(pkg, n, k):
    P = bi.make_problem(n, seed=n + k)
    A, B = problem_on_device(P)
    W = to_dev(bi.start_block(n, k, 8))
    lam = torch.linspace(0.5, 4.0, k, dtype=torch.float64, device="cuda")
    X, Y = W[:, :n], W[:, n:]
    R = torch.cat([X @ A.T + Y @ B.T, -(X @ B.conj().T) - (Y @ A.conj().T)], 1) - lam[:, None] * W
    ref = torch.linalg.vector_norm(R, dim=1).cpu().numpy()
    np.testing.assert_allclose(pkg.residuals(A, B, W, lam).cpu().numpy(), ref, rtol=1e-12)
    W[3, 5] = float("nan")
    got = pkg.residuals(A, B, W, lam).cpu().numpy()
    assert np.isnan(got[3]) and np.isfinite(np.delete(got, 3)).all()
    A[7, 7] = float("nan")
    assert np.isnan(pkg.residuals(A, B, W, lam).cpu().numpy()).all()


def test_residuals_over_blocks_of_rows(pkg):
    """n = 6144: the digits of H are cut into two blocks of rows."""
    n, k = 6144, 3
    g = torch.Generator(device="cuda").manual_seed(2)
    A = torch.randn((n, n), generator=g, dtype=torch.complex128, device="cuda")
    B = torch.randn((n, n), generator=g, dtype=torch.complex128, device="cuda")
    W = torch.randn((k, 2 * n), generator=g, dtype=torch.complex128, device="cuda")
    lam = torch.linspace(0.5, 4.0, k, dtype=torch.float64, device="cuda")
    X, Y = W[:, :n], W[:, n:]
    R = torch.cat([X @ A.T + Y @ B.T, -(X @ B.conj().T) - (Y @ A.conj().T)], 1) - lam[:, None] * W
    ref = torch.linalg.vector_norm(R, dim=1).cpu().numpy()
    np.testing.assert_allclose(pkg.residuals(A, B, W, lam).cpu().numpy(), ref, rtol=1e-12)
