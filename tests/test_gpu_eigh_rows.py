"""The FP64 Jacobi at the row counts where its V pass changes the rows of a CTA (152 and 304 on
a GB300), and the FP32 block Jacobi on matrices of which few block pairs, or none, rotate."""
import numpy as np
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


def _check(pkg, G, method):
    # the tolerances of tests/test_gpu_eigh.py
    k = G.shape[0]
    theta, V = pkg.eigh(torch.from_numpy(G).cuda(), method=method, thr=2e-16)
    theta, V = theta.cpu().numpy(), V.cpu().numpy()
    nrm = np.linalg.norm(G, 2)
    assert np.abs(np.sort(theta) - np.linalg.eigvalsh(G)).max() <= 1e-12 * nrm
    assert np.linalg.norm(G @ V - V * theta, axis=0).max() <= (1e-12 + 1e-13 * np.sqrt(k)) * nrm
    assert np.abs(V.conj().T @ V - np.eye(k)).max() <= 1e-12


def _hermitian(k, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((k, k)) + 1j * rng.standard_normal((k, k))
    return (X + X.conj().T) / 2


@pytest.mark.parametrize("k", [2, 150, 152, 154, 304, 306])
def test_jacobi_rows_per_cta(pkg, k):
    _check(pkg, _hermitian(k, k), "jacobi")


@pytest.mark.parametrize("pairs", [0, 1, 40])
def test_mixed_with_few_coupled_blocks(pkg, pairs):
    k = 288
    rng = np.random.default_rng(pairs)
    G = np.diag(np.linspace(1.0, 40.0, k)).astype(np.complex128)
    for _ in range(pairs):
        i, j = rng.choice(k, 2, replace=False)
        G[i, j] += 0.3 + 0.1j
        G[j, i] = np.conj(G[i, j])
    _check(pkg, G, "mixed")
