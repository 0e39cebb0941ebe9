"""The precision form's FP32 row Jacobi on blocks of rows, through its truncated
SVD with nothing truncated (the FP32 solve then runs on the r x c matrix): row
counts around the block size and its smallest use, columns around the edges of
every register variant (256, 512, 1024, 2048, 4096) and beyond.

Tolerances: U and X come from FP64-accurate products (2^-42 |row| |column|),
U ends orthonormal to 1e-10 and the kept block meets the form's bar of 1e-7
whatever basis the FP32 solve hands over."""
import numpy as np
import pytest

from paper_2003_13163_gb300.circuits import random_complex
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    return need_gpu()


@pytest.mark.parametrize("r,c", [(31, 64), (32, 255), (33, 257), (35, 512), (36, 513), (37, 1025), (40, 2048),
                                 (41, 2049), (34, 4097), (130, 130)])
def test_quad_jacobi_sizes(M, r, c):
    import torch
    U0 = np.linalg.qr(random_complex((r, r), r))[0]
    V0 = np.linalg.qr(random_complex((c, r), c + 1))[0]
    s = np.exp(-np.linspace(0, 9, r))
    A = (U0 * s) @ V0.conj().T
    U, X, lam2 = M.svd_truncated(torch.tensor(A, device="cuda"), r, "mixed")
    U, X = U.cpu().numpy(), X.cpu().numpy()
    assert len(lam2) == r
    assert np.linalg.norm(U @ X - A) <= 1e-7 * np.linalg.norm(A)
    assert np.abs(U.conj().T @ U - np.eye(r)).max() < 1e-10
    np.testing.assert_allclose(lam2, s ** 2, rtol=0, atol=1e-11)
