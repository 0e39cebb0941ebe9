"""The precision form on a block whose FP32 copy has no nonzero row norm: the
FP32 selection orders all directions, none of which is above another. The zero
matrix gives one kept direction of weight zero; a block whose squared entries
are below the FP32 range (1e-25) is solved by the FP64 step alone.

Tolerance: 1e-10 of the largest value, the form's bar for an untruncated block."""
import numpy as np
import pytest

from paper_2003_13163_gb300.circuits import random_complex
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu
SIZES = [(1, 1), (8, 9), (31, 31), (33, 40), (100, 130), (256, 256)]


@pytest.fixture(scope="module")
def M():
    return need_gpu()


def factor(M, A):
    import torch
    U, X, lam2 = M.svd_truncated(torch.tensor(A, device="cuda"), A.shape[0], "mixed")
    return U.cpu().numpy(), X.cpu().numpy(), lam2


@pytest.mark.parametrize("r,c", SIZES)
def test_zero_matrix(M, r, c):
    U, X, lam2 = factor(M, np.zeros((r, c), dtype=np.complex128))
    assert list(lam2) == [0.0] and np.abs(X).max() == 0.0
    assert abs(np.linalg.norm(U) - 1.0) < 1e-10


@pytest.mark.parametrize("r,c", SIZES)
def test_below_fp32_range(M, r, c):
    B = random_complex((r, c), r)
    s = np.linalg.svd(B, compute_uv=False)
    U, X, lam2 = factor(M, B * 1e-25)
    assert len(lam2) == r
    assert np.abs(np.sqrt(lam2) * 1e25 - s).max() < 1e-10 * s[0]
    assert np.linalg.norm(U @ (X * 1e25) - B) < 1e-10 * np.linalg.norm(B)
    assert np.abs(U.conj().T @ U - np.eye(r)).max() < 1e-10
