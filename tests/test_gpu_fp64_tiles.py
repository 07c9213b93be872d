"""The FP64 H application and complex GEMM at the edges of their tiles (32 rows, 8 to 64
columns) and K splits, through the residual and Rayleigh-Ritz entry points."""
import numpy as np
import pytest
import torch

import bse_inputs as bi
from oracle import rayleigh_ritz as orr
from tests.gpu_util import problem_on_device, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2601_10557_gb300 as p
    p.lib()
    return p


# each output is a sum of 2n products: |error| <= 2n * 2^-53 * (a few) of |H| |w|, far below
# 1e-12 of the residual's norm (of the order of |H| |w| for these random vectors)
@pytest.mark.parametrize("n,k", [(1, 1), (2, 3), (31, 1), (32, 8), (33, 9), (64, 6), (65, 31), (97, 33), (160, 65)])
def test_residuals_at_tile_edges(pkg, n, k):
    P = bi.make_problem(n, seed=n + 7 * k)
    A, B = problem_on_device(P)
    W = bi.start_block(n, k, 8).T
    lam = np.linspace(0.5, 4.0, k)
    ref = orr.residuals(P.A, P.B, W, lam)
    lam_d = torch.from_numpy(lam).cuda()
    got = pkg.residuals(A, B, to_dev(W.T), lam_d).cpu().numpy()
    np.testing.assert_allclose(got, ref, rtol=1e-12)
    from paper_2601_10557_gb300._lib import residuals_noalloc
    out = torch.empty(k, dtype=torch.float64, device="cuda")
    residuals_noalloc(A, B, to_dev(W.T), lam_d, out)
    np.testing.assert_allclose(out.cpu().numpy(), ref, rtol=1e-12)
