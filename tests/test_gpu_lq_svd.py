"""The LQ-preconditioned truncated SVD of the FP64 form at the edges of its
variants: the smallest row count that takes it and one below, rows in
registers up to 256 and 1024 columns and streamed beyond, more rows than
CTAs, zero and repeated rows.

Tolerances: r Householder steps and at most 40 sweeps of r - 1 rotations per
row, each unitary to a few eps: 10 eps sqrt(41 r) for U, and for the rows of
X relative to their own norm (they are sigma times an orthonormal row)."""
import numpy as np
import pytest

from paper_2003_13163_gb300.circuits import random_complex
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu
EPS = 2.2e-16


@pytest.fixture(scope="module")
def M():
    return need_gpu()


def check(M, A, rank):
    import torch
    r, c = A.shape
    U, X, lam2 = M.svd_truncated(torch.tensor(A, device="cuda"), r, "fp64")
    U, X = U.cpu().numpy(), X.cpu().numpy()
    ref = np.linalg.svd(A, compute_uv=False)
    tol = 10 * EPS * np.sqrt(41 * r)
    assert len(lam2) == rank
    assert np.abs(U.conj().T @ U - np.eye(rank)).max() < tol
    n = np.sqrt(lam2)
    G = (X @ X.conj().T) / np.outer(n, n)
    assert np.abs(G - np.eye(rank)).max() < tol * np.sqrt(c)
    assert np.abs(U @ X - A).max() <= tol * ref[0]
    assert np.abs(n - ref[:rank]).max() <= tol * ref[0]


@pytest.mark.parametrize("r,c", [(7, 30), (8, 8), (8, 256), (9, 257), (64, 256), (129, 130), (30, 1024), (30, 1025),
                                 (500, 520)])
def test_lq_svd_sizes(M, r, c):
    check(M, random_complex((r, c), seed=r + c) * np.exp(-np.linspace(0, 9, c))[None, :], r)


def test_lq_svd_small_singular_values(M):
    """Eleven decades: every kept factor stays orthonormal."""
    U = np.linalg.qr(random_complex((40, 40), 3))[0]
    V = np.linalg.qr(random_complex((90, 40), 4))[0]
    check(M, (U * 10.0 ** -np.linspace(0, 11, 40)) @ V.conj().T, 40)


def test_lq_svd_rank_deficient(M):
    A = random_complex((20, 6), 1) @ random_complex((6, 50), 2)
    A[7] = 0
    A[11] = A[3]
    A[0] = 0
    check(M, A, 6)
