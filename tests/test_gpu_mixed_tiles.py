"""The tensor-core filter at the edges of its output tiles (256 rows of the real form, column
tiles of 32 to 256), of its K blocks (64) and of its schedule (K ranges of tiles, full waves of
CTA pairs followed by cut tiles), against the FP64 filter of the library."""
import numpy as np
import pytest
import torch

import bse_inputs as bi
from tests.gpu_util import problem_on_device, to_dev

pytestmark = pytest.mark.gpu

# the filter gates of FP32-class and 16-bit pieces (tests/test_gpu_mixed.py)
TOL = {"fp16x3": 1e-5, "bf16x6": 1e-5, "bf16x3": 6e-5}


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2601_10557_gb300 as p
    if not p.has_mixed():
        pytest.fail("tensor-core filter not available on this device")
    return p


def _device_problem(n, seed):
    """A hermitian positive A and a small symmetric B made on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn((n, n), generator=g, dtype=torch.complex128, device="cuda")
    A = (X + X.conj().T) * (0.5 / np.sqrt(n)) + 5.0 * torch.eye(n, dtype=torch.complex128, device="cuda")
    Y = torch.randn((n, n), generator=g, dtype=torch.complex128, device="cuda")
    return A.contiguous(), ((Y + Y.T) * (0.05 / np.sqrt(n))).contiguous()


@pytest.mark.parametrize("precision", ["fp16x3", "bf16x6", "bf16x3"])
# rows 2n: 2, 62 / 64 / 66 around a K block, 254 / 256 / 258 around a tile; columns 2k around
# 32, 160 (one or two x0 y0 buffers) and 256
@pytest.mark.parametrize("n,k", [(1, 1), (31, 2), (32, 15), (33, 16), (127, 17), (128, 80), (129, 81), (300, 128),
                                 (257, 129)])
def test_filter_at_tile_edges(pkg, precision, n, k):
    P = bi.make_problem(n, seed=3 * n + k)
    A, B = problem_on_device(P)
    degs = 1 + np.arange(k) % 4
    W = to_dev(bi.start_block(n, k, 5))
    mus = (0.5 * float(P.d.min()), 0.8 * float(P.d.max()) + 0.1, 1.5 * float(P.d.max()))
    ref = pkg.filter(A, B, W.clone(), degs, *mus, precision="fp64")
    got = pkg.filter(A, B, W.clone(), degs, *mus, precision=precision)
    assert torch.linalg.vector_norm(got - ref) <= TOL[precision] * torch.linalg.vector_norm(ref)


# 96 tiles: one full wave of 76 pairs and 20 tiles in three K ranges each; 176 tiles: two waves
# and 24 tiles; the ragged degrees end in narrow launches of few columns
@pytest.mark.parametrize("n,k", [(2048, 700), (2050, 1290)])
def test_filter_over_full_waves(pkg, n, k):
    A, B = _device_problem(n, k)
    degs = np.where(np.arange(k) < 9, 3, 1 + np.arange(k) % 2)
    g = torch.Generator(device="cuda").manual_seed(n)
    W = torch.randn((k, 2 * n), generator=g, dtype=torch.complex128, device="cuda")
    ref = pkg.filter(A, B, W.clone(), degs, 1.5, 4.0, 8.0, precision="fp64")
    got = pkg.filter(A, B, W.clone(), degs, 1.5, 4.0, 8.0, precision="fp16x3")
    again = pkg.filter(A, B, W.clone(), degs, 1.5, 4.0, 8.0, precision="fp16x3")
    assert torch.linalg.vector_norm(got - ref) <= 1e-5 * torch.linalg.vector_norm(ref)
    assert torch.equal(got, again)  # the K ranges are summed in a fixed order
