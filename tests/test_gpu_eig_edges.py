"""Pivoted Cholesky and one-sided Jacobi at the sizes where their kernels change."""

import numpy as np
import pytest
import torch

import paper_2503_18056_gb300 as T

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52


def graded(n, rank, seed):
    g = np.random.default_rng(seed)
    B = g.standard_normal((rank, n)) * np.geomspace(1.0, 1e-5, rank)[:, None]
    return B.T @ B


# a warp's entries per row change at multiples of 32, the cluster's warps per CTA at
# multiples of 32 rows, the solver at 256 and the factorisation at 608
@pytest.mark.parametrize("n", [1, 2, 3, 31, 32, 33, 64, 65, 96, 97, 128, 129, 160, 161, 192, 193, 224, 225, 255, 256,
                               257, 608, 609])
@pytest.mark.parametrize("full", [True, False])
def test_syev_psd_and_pchol(n, full):
    rank = n if full else max(1, n // 2)
    K = graded(n, rank, n)
    W, k = T.pchol(torch.tensor(K, device="cuda"))
    assert 1 <= k <= n
    W = W.cpu().numpy()
    # each residual entry: k products and the pivots left out, both relative to
    # the largest diagonal entry
    assert np.abs(W.T @ W - K).max() <= 4 * (n + 1) * EPS * np.abs(np.diag(K)).max()
    lam, V, _ = T.syev_psd(torch.tensor(K, device="cuda"))
    lam, V = lam.cpu().numpy(), V.cpu().numpy()
    assert np.all(np.diff(lam) <= 0) and lam[-1] >= 0
    # factorisation and at most about 12 n rotations of a row, each a few roundings
    tol = 64 * (n + 1) * EPS * lam[0]
    assert np.abs(lam - np.linalg.eigvalsh(K)[::-1]).max() <= tol
    assert np.abs((V.T * lam) @ V - K).max() <= tol
    U = V[lam > 0]
    # unit rows, orthogonal to the skip threshold sqrt(n) eps and the rounding of the product
    assert np.abs(U @ U.T - np.eye(len(U))).max() <= 8 * (n + 1) * EPS


# pairs of a CTA (four warps a pair up to twice the SMs' rows, then two), the grid
# kernel's longest rows and the streaming kernel above them
@pytest.mark.parametrize("n,rank", [(304, 304), (305, 305), (700, 300), (1024, 1024), (1024, 500), (1025, 1025), (1100, 1050)])
def test_syev_psd_between_the_grid_kernels(n, rank):
    K = graded(n, rank, n)
    lam, V, _ = T.syev_psd(torch.tensor(K, device="cuda"))
    lam, V = lam.cpu().numpy(), V.cpu().numpy()
    tol = 64 * (n + 1) * EPS * lam[0]
    assert np.all(np.diff(lam) <= 0) and lam[-1] >= 0
    assert np.abs(lam - np.linalg.eigvalsh(K)[::-1]).max() <= tol
    assert np.abs((V.T * lam) @ V - K).max() <= tol
    U = V[lam > 0]
    assert np.abs(U @ U.T - np.eye(len(U))).max() <= 8 * (n + 1) * EPS


def test_captured_eigensolves_below_a_capacity_above_the_grid_kernel():
    """Cap 210 in 2D: 1,051 grown columns, so a captured step launches all three
    kernels and each size takes the host path's."""
    import workloads

    p = workloads.problem("small_2d", n=(32, 30), n_theta=16, n_phi=32, eps=1e-6, bc=1)
    p["max_rank"] = 210
    a, b = T.TTSN.from_problem(p), T.TTSN.from_problem(p)
    b.set_graph(True)
    for _ in range(5):
        assert a.step()["ranks"] == b.step()["ranks"]
    assert 5 * a.ranks()[1] + 1 > 256
    for x, y in zip(a.cores(), b.cores()):
        assert torch.equal(torch.as_tensor(x), torch.as_tensor(y))
