"""The split product's K parts (products with fewer tiles than SMs) and its tile
orders: one tile with a short and a long inner dimension, a remainder in the
parts, more tiles than one group of 16 row blocks, and a repeated call (the
per-tile counters are reset by the kernel).

Bounds as in test_gpu_ozgemm: 1e-11 |A| |B| element-wise; the parts' sums are
added in FP64 in a fixed order, so two calls give the same bits."""
import numpy as np
import pytest

from paper_2003_13163_gb300.circuits import random_complex
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    return need_gpu()


@pytest.mark.parametrize("m,n,k", [(100, 20, 16), (64, 64, 319), (64, 64, 320), (128, 32, 2000), (130, 33, 1111), (64, 700, 2048),
                                   (513, 300, 1100), (1100, 500, 300), (2200, 130, 40)])
def test_split_parts(M, m, n, k):
    import torch
    A, B = random_complex((m, k), seed=m + k), random_complex((k, n), seed=n + k + 1)
    At, Bt = torch.tensor(A, device="cuda"), torch.tensor(B, device="cuda")
    C = M.gemm_ex(At, Bt, 0, 0, "fp64", 1)
    assert torch.equal(C, M.gemm_ex(At, Bt, 0, 0, "fp64", 1))
    assert np.all(np.abs(C.cpu().numpy() - A @ B) <= 1e-11 * (np.abs(A) @ np.abs(B)))
