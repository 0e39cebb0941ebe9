"""The precision form ends with MPO_ERR_NOCONV, not with a success code and
factors of NaN, when a matrix holds infinities or NaN: where nothing is
truncated (the FP32 solve runs on the matrix) and after the subspace iteration."""
import numpy as np
import pytest

from paper_2003_13163_gb300.circuits import random_complex
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("r,cap", [(8, 8), (33, 33), (64, 64), (130, 130), (130, 20)])
def test_refused(r, cap, value):
    import torch
    M = need_gpu()
    A = random_complex((r, r + 1), 1)
    A[r // 2, 3] = value
    with pytest.raises(M.MPOError) as e:
        M.svd_truncated(torch.tensor(A, device="cuda"), cap, "mixed")
    assert e.value.code == -4
