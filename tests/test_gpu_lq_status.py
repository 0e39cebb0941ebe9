"""A wait that runs out in the LQ step alone is reported.

32 rows of a million columns: a Householder step streams whole rows while the
CTAs whose rows are done wait at its barrier, several hundred microseconds; the
solves that follow work on 32 x 32 and wait a few. A limit of 100 us is met
by the first kernel only. The kernel leaves with its status word, nothing faults."""
import numpy as np
import pytest

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def test_lq_timeout_is_reported():
    import torch
    M = need_gpu()
    g = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randn((32, 1000000), dtype=torch.complex128, device="cuda", generator=g)
    with pytest.raises(M.MPOError) as e:
        M.svd_truncated(A, 8, "fp64", barrier_timeout_s=1e-4)
    assert e.value.code == -5
    # with the default limit the same call gives the factorisation
    U, X, lam2 = M.svd_truncated(A, 8, "fp64")
    ref = torch.linalg.eigvalsh(A @ A.conj().T).cpu().numpy()[::-1][:8]
    np.testing.assert_allclose(lam2, ref, rtol=1e-10)
    assert float((U.conj().T @ A - X).abs().max()) <= 1e-10 * float(A.abs().max())
