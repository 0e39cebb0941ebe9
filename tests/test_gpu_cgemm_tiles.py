"""The SIMT complex128 product at the edges of its two tile sizes (8 x 8 with a
four-way split of k below 152 tiles of 16 x 16, 16 x 16 above), in every
operand form.

Tolerance: K products and additions of relative error eps each, against
NumPy's own: 4 eps K |A| |B| element-wise."""
import numpy as np
import pytest

from paper_2003_13163_gb300.circuits import random_complex
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    return need_gpu()


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (8, 8, 8), (9, 7, 33), (17, 15, 31), (64, 64, 100), (176, 224, 16),
                                   (161, 250, 47), (2500, 16, 65)])
@pytest.mark.parametrize("opA,opB", [(0, 0), (1, 0), (0, 1), (1, 1)])
def test_cgemm_tiles(M, m, n, k, opA, opB):
    import torch
    A, B = random_complex((m, k), seed=m + k), random_complex((k, n), seed=n + k + 1)
    At = torch.tensor(A.conj().T.copy() if opA else A, device="cuda")
    Bt = torch.tensor(B.conj().T.copy() if opB else B, device="cuda")
    C = M.gemm_ex(At, Bt, opA, opB, "fp64", engine=0).cpu().numpy()
    assert np.all(np.abs(C - A @ B) <= 4 * 2.2e-16 * k * (np.abs(A) @ np.abs(B)))
