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


@pytest.fixture(scope="module")
def tensor_cores(pkg):
    if not pkg.has_mixed():
        pytest.fail("tensor-core filter not available on this device")
    return pkg


# The tensor-core filters' gates of a whole vector (tests/test_gpu_mixed.py, test_gpu_h2.py) for each
# half: FP16x3 keeps 22 bits of an operand entry down to 2^-11 of the largest of its row or vector
# (16-bit pieces of 11 bits each from 2^13 down to 2^-24), so down to a coupling of 1e-4 (2^-13.3)
# all but two of them; the BF16 pieces have FP32's exponent range.
TOL = {"fp16x3": 1e-5, "bf16x6": 1e-5, "bf16x3": 6e-5}


@pytest.mark.parametrize("precision", ["fp16x3", "bf16x6", "bf16x3"])
@pytest.mark.parametrize("beta", [0.3, 1e-3, 1e-4])
# operand rows n around a tile of 256 rows, columns 4k around 32, 160 and 256, K = 4n around a
# block of 64; (300, 70): K ranges, (640, 24)
@pytest.mark.parametrize("n,k,deg", [(31, 1, 3), (47, 8, 4), (129, 33, 4), (255, 9, 3), (256, 40, 3),
                                     (257, 41, 3), (300, 70, 4), (640, 24, 4), (900, 400, 2), (520, 700, 2)])
def test_tensor_core_filter_keeps_both_halves(tensor_cores, precision, n, k, deg, beta):
    P = bi.make_problem(n, seed=n + k, beta=beta)
    A, B = problem_on_device(P)
    W = _block(n, k, 4, beta)
    mus = (0.5 * float(P.d.min()), 0.8 * float(P.d.max()) + 0.1, 1.5 * float(P.d.max()))
    ref = _filter(A, B, W, deg, *mus)
    got = tensor_cores.filter(A, B, W.clone(), [deg] * k, *mus, precision=precision)
    assert max(_errors(got, ref)) <= TOL[precision]


@pytest.mark.parametrize("beta", [0.3, 1e-3])
@pytest.mark.parametrize("n,k", [(64, 9), (300, 70)])
def test_explicit_square_filter_keeps_both_halves(tensor_cores, n, k, beta):
    P = bi.make_problem(n, seed=n + k, beta=beta)
    A, B = problem_on_device(P)
    W = _block(n, k, 4, beta)
    mus = (0.5 * float(P.d.min()), 0.8 * float(P.d.max()) + 0.1, 1.5 * float(P.d.max()))
    ref = _filter(A, B, W, 4, *mus)
    got = tensor_cores.filter_h2(A, B, W.clone(), [4] * k, *mus)
    assert max(_errors(got, ref)) <= 5e-5


# full waves of CTA pairs and K ranges of the tiles left over, ragged degrees; ranges that cross
# from one tile into the next behind none (1100, 250), (1270, 500), one (2048, 900) and two
# (2048, 1500) full waves
@pytest.mark.parametrize("n,k", [(2048, 700), (2050, 645), (1100, 250), (1270, 500), (2048, 900), (2048, 1500)])
def test_tensor_core_filter_halves_over_full_waves(tensor_cores, n, k):
    g = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randn((n, n), generator=g, dtype=torch.complex128, device="cuda")
    A = (X + X.conj().T) * (0.5 / np.sqrt(n)) + 5.0 * torch.eye(n, dtype=torch.complex128, device="cuda")
    Y = torch.randn((n, n), generator=g, dtype=torch.complex128, device="cuda")
    B = (Y + Y.T) * (1e-3 / np.sqrt(n))
    W = torch.randn((k, 2 * n), generator=g, dtype=torch.complex128, device="cuda")
    W[:, n:] *= 1e-3
    degs = np.where(np.arange(k) < 9, 3, 1 + np.arange(k) % 2)
    got = tensor_cores.filter(A, B, W.clone(), degs, 1.5, 4.0, 8.0, precision="fp16x3")
    again = tensor_cores.filter(A, B, W.clone(), degs, 1.5, 4.0, 8.0, precision="fp16x3")
    assert torch.equal(got, again)  # the K ranges are summed in a fixed order
    for d in (1, 2, 3):
        sel = torch.from_numpy(np.flatnonzero(degs == d)).cuda()
        assert max(_errors(got[sel], _filter(A, B, W[sel], d, 1.5, 4.0, 8.0))) <= 1e-5
