"""Each half of a filtered vector is accurate relative to its own size.  With a weak coupling B
(and in the solver's start block) the lower half is orders of magnitude smaller than the upper
one, and a user of the vectors reads it by itself; the norm of the whole vector does not show
its error."""
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
    p.lib()
    return p


def _hop(A, B, W):
    n = A.shape[0]
    X, Y = W[:, :n], W[:, n:]
    return torch.cat([X @ A.T + Y @ B.T, -(X @ B.conj().T) - (Y @ A.conj().T)], 1)


def _filter(A, B, W, deg, mu1, mune, muN):
    """The recurrence in plain 64-bit products, each half summed by itself."""
    c, e = 0.5 * (mune ** 2 + muN ** 2), 0.5 * (muN ** 2 - mune ** 2)
    s1 = e / (mu1 ** 2 - c)
    prev, cur, sig = None, W, s1
    for j in range(deg):
        T = _hop(A, B, _hop(A, B, cur)) - c * cur
        if j == 0:
            prev, cur = cur, (s1 / e) * T
        else:
            sn = 1.0 / (2.0 / s1 - sig)
            prev, cur = cur, (2.0 * sn / e) * T - sig * sn * prev
            sig = sn
    return cur


def _block(n, k, seed, lower):
    W = to_dev(bi.start_block(n, k, seed))
    W[:, n:] *= lower / float(W[:, n:].abs().max() / W[:, :n].abs().max())
    return W


def _errors(got, ref):
    n = ref.shape[1] // 2
    return [float(torch.linalg.vector_norm(g - r) / torch.linalg.vector_norm(r))
            for g, r in ((got[:, :n], ref[:, :n]), (got[:, n:], ref[:, n:]))]


# A half is a sum of 2n products in each of 2 deg applications of H, and the recurrence scales
# all of them alike: 2 deg sqrt(2n) 2^-53 times a small factor, far below the FP64 filter's gate
# of 1e-12 (tests/test_gpu_parity.py), which a lower half known to 2^-53 of the upper one misses
# by three orders of magnitude at a coupling of 1e-6.
@pytest.mark.parametrize("beta", [0.3, 1e-3, 1e-6])
@pytest.mark.parametrize("n,k,deg", [(31, 1, 3), (64, 9, 8), (129, 33, 5), (512, 30, 8)])
def test_fp64_filter_keeps_both_halves(pkg, n, k, deg, beta):
    P = bi.make_problem(n, seed=n + k, beta=beta)
    A, B = problem_on_device(P)
    W = _block(n, k, 4, beta)
    mus = (0.9 * float(P.d.min()), 0.5 * float(P.d.max()) + 0.5, 1.1 * float(P.d.max()))
    ref = _filter(A, B, W, deg, *mus)
    got = pkg.filter(A, B, W.clone(), [deg] * k, *mus)
    assert max(_errors(got, ref)) <= 1e-12
    # the half that is small may also be the upper one
    swap = lambda V: torch.cat([V[:, n:], V[:, :n]], 1).conj().resolve_conj()
    got = pkg.filter(A, B, swap(W), [deg] * k, *mus)
    assert max(_errors(swap(got), ref)) <= 1e-12


def test_fp64_filter_without_coupling_keeps_a_zero_half(pkg):
    """B = 0 and y = 0: the lower half is a sum of zeros."""
    n, k = 130, 12
    P = bi.make_problem(n, seed=3, b_zero=True)
    A, B = problem_on_device(P)
    W = to_dev(bi.start_block(n, k, 4))
    W[:, n:] = 0.0
    got = pkg.filter(A, B, W, [4] * k, 0.9 * float(P.d.min()), 5.0, 1.1 * float(P.d.max()))
    assert not bool(torch.any(got[:, n:] != 0.0)) and bool(torch.all(torch.isfinite(got.abs())))
