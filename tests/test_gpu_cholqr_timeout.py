"""A grid barrier that runs out in the precision form's Cholesky QR: the launches
of the same factorisation that follow leave at once, the call returns
MPO_ERR_TIMEOUT and the next one is unaffected. The products run on the SIMT
kernels (tensor_cores = -1), which wait for nothing."""
import ctypes

import numpy as np
import pytest

from paper_2003_13163_gb300.circuits import random_complex
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def call(M, A, cap, limit):
    import torch
    r, c = A.shape
    o = M.default_opts()
    o.tensor_cores = -1
    o.barrier_timeout_s = limit
    A = torch.tensor(A, device="cuda")
    U = torch.zeros((r, cap), dtype=A.dtype, device="cuda")
    X = torch.zeros((cap, c), dtype=A.dtype, device="cuda")
    lam2, k = np.zeros(cap), ctypes.c_int()
    torch.cuda.synchronize()
    rc = M.load_library().mpo_svd_truncated(r, c, A.data_ptr(), cap, M.PRECISIONS["mixed"], ctypes.byref(o), U.data_ptr(),
                                            X.data_ptr(), lam2.ctypes.data_as(ctypes.POINTER(ctypes.c_double)),
                                            ctypes.byref(k), None)
    return rc, lam2


def test_timeout_then_normal_call():
    M = need_gpu()
    A = random_complex((300, 320), 1) * np.exp(-np.linspace(0, 9, 320))
    assert call(M, A, 70, 1e-9)[0] == -5
    rc, lam2 = call(M, A, 70, 0.0)
    assert rc == 0
    s = np.linalg.svd(A, compute_uv=False)
    np.testing.assert_allclose(lam2, s[:70] ** 2, rtol=0, atol=1e-11 * s[0] ** 2)
