"""The gradient products where only the lower triangle is computed (n >= 1088 on a GB300):
against the same formula in plain FP64, with exact symmetry, around the rule and with sizes
that fit no tile."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2601_10557_gb300 as p
    p.lib()
    return p


@pytest.mark.parametrize("n,nev", [(1087, 3), (1088, 3), (1089, 40), (1153, 7), (2047, 25)])
def test_gradient_triangle(pkg, n, nev):
    g = torch.Generator(device="cuda").manual_seed(n)
    V = torch.randn((nev, 2 * n), generator=g, dtype=torch.complex128, device="cuda")
    V[:, n:] *= 0.1
    V = V / torch.linalg.vector_norm(V, dim=1, keepdim=True)
    w = torch.randn(nev, generator=g, dtype=torch.float64, device="cuda")
    gA, gB = pkg.grad(V, w)
    X, Y = V[:, :n], V[:, n:]
    c = w / (X.abs().square().sum(1) - Y.abs().square().sum(1))
    refA = (X.T * c) @ X.conj() + (Y.conj().T * c) @ Y
    refB = (X.T * c) @ Y.conj() + (Y.conj().T * c) @ X
    # 4 nev products a sum, each to FP64 rounding
    assert torch.linalg.vector_norm(gA - refA) <= 1e-13 * torch.linalg.vector_norm(refA)
    assert torch.linalg.vector_norm(gB - refB) <= 1e-13 * torch.linalg.vector_norm(refB)
    off = ~torch.eye(n, dtype=torch.bool, device="cuda")
    if n >= 1088:
        assert torch.equal(gA.conj().T[off], gA[off])
        assert torch.equal(gB.T[off], gB[off])
