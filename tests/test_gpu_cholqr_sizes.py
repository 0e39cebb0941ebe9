"""The precision form's truncated SVD at subspace sizes around the 64-row tiles
of its Cholesky factorisation (m = cap + oversample = 2 cap by default): one
tile, a tile more or less, a single row, several tiles with a ragged one.

Tolerances: the products carry 2^-42 |row| |column| and the left factor ends
with Newton-Schulz steps on them, so U is orthonormal to 1e-10; the kept block
meets the form's bar of 1e-7."""
import numpy as np
import pytest

from paper_2003_13163_gb300.circuits import random_complex
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    return need_gpu()


@pytest.mark.parametrize("r,c,cap", [(40, 40, 1), (140, 140, 31), (140, 141, 32), (140, 150, 33), (300, 310, 64),
                                     (300, 300, 65), (700, 720, 161)])
def test_mixed_svd_tile_edges(M, r, c, cap):
    import torch
    U0 = np.linalg.qr(random_complex((r, r), r))[0]
    V0 = np.linalg.qr(random_complex((c, r), c + 1))[0]
    s = np.exp(-6.9 * (np.arange(r) / max(cap, 4)) ** 0.52)
    A = (U0 * s) @ V0.conj().T
    U, X, lam2 = M.svd_truncated(torch.tensor(A, device="cuda"), cap, "mixed")
    U, X = U.cpu().numpy(), X.cpu().numpy()
    ref = (U0[:, :cap] * s[:cap]) @ V0[:, :cap].conj().T
    assert np.linalg.norm(U @ X - ref) <= 1e-7 * np.linalg.norm(ref)
    assert np.abs(U.conj().T @ U - np.eye(U.shape[1])).max() < 1e-10
    np.testing.assert_allclose(lam2, s[:cap] ** 2, rtol=1e-9, atol=1e-14)
