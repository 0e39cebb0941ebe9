"""Blocks scaled towards the end of the FP64 range, on every route of the row
solver (fewer than 8 rows, the LQ step, its FP32 start): the factorisation is
accurate while the squares of the entries are normal numbers, and refused with
MPO_ERR_NOCONV, not wrong, when they are not. Rows far below the others
change nothing.

Tolerance: as for the sizes at scale 1, 10 eps sqrt(41 r) of the largest."""
import numpy as np
import pytest

from paper_2003_13163_gb300.circuits import random_complex
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu
SIZES = [(6, 9), (20, 50), (64, 70)]


@pytest.fixture(scope="module")
def M():
    return need_gpu()


def factor(M, A):
    import torch
    U, X, lam2 = M.svd_truncated(torch.tensor(A, device="cuda"), A.shape[0], "fp64")
    return U.cpu().numpy(), X.cpu().numpy(), lam2


@pytest.mark.parametrize("r,c", SIZES)
@pytest.mark.parametrize("scale", [1e-145, 1e-130, 1.0, 1e150])
def test_scaled(M, r, c, scale):
    B = random_complex((r, c), r)
    U, X, lam2 = factor(M, B * scale)
    s = np.linalg.svd(B, compute_uv=False)
    tol = 10 * 2.2e-16 * np.sqrt(41 * r) * s[0]
    assert len(lam2) == r
    assert np.abs(np.sqrt(lam2) / scale - s).max() < tol
    assert np.abs(U @ (X / scale) - B).max() < tol
    assert np.abs(U.conj().T @ U - np.eye(r)).max() < tol / s[0]


@pytest.mark.parametrize("r,c", SIZES)
@pytest.mark.parametrize("scale", [1e-152, 1e-153, 1e-155, 1e-158, 1e-160])
def test_too_small_is_refused(M, r, c, scale):
    with pytest.raises(M.MPOError) as e:
        factor(M, random_complex((r, c), r) * scale)
    assert e.value.code == -4


@pytest.mark.parametrize("r,c", SIZES)
def test_negligible_rows(M, r, c):
    B = random_complex((r, c), r)
    B[1::3] *= 1e-158
    U, X, lam2 = factor(M, B)
    s = np.linalg.svd(B, compute_uv=False)
    k = r - len(B[1::3])
    tol = 10 * 2.2e-16 * np.sqrt(41 * r) * s[0]
    assert len(lam2) == k and np.abs(np.sqrt(lam2) - s[:k]).max() < tol
    assert np.abs(U @ X - B).max() < tol
    U, X, lam2 = factor(M, np.zeros((r, c), dtype=np.complex128))
    assert np.abs(X).max() == 0 and lam2.sum() == 0
