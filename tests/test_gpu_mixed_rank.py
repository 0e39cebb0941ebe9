"""Truncated blocks whose rank, to the precision form's resolution, is below the
directions that its FP64 step carries (cap + 64): the values and couplings of
the directions beyond it are rounding, of which no correction may be made.

Tolerances are the form's: U orthonormal to 1e-10, the kept block within 1e-7 of
|A|, squared values to 1e-11 of the largest. Spectra keep 10 % away from the
cutoff of 1e-7, where the form resolves values to a percent."""
import numpy as np
import pytest

from paper_2003_13163_gb300.circuits import random_complex
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def orthonormal(n, k, seed):
    return np.linalg.qr(random_complex((n, k), seed))[0]


def decay(r, c):     # 10^(-0.12 j): 1.10e-7 at j = 58, 0.83e-7 at j = 59
    return (orthonormal(r, r, 1) * 10.0 ** (-0.12 * np.arange(r))) @ orthonormal(c, r, 2).conj().T


BLOCKS = {
    "rank": lambda r, c: random_complex((r, r // 4), 3) @ random_complex((r // 4, c), 4),
    "decay": decay,
    "decaying_rows": lambda r, c: 10.0 ** (-0.12 * np.arange(r))[:, None] * orthonormal(c, r, 5).conj().T,
}


@pytest.mark.parametrize("r,c,cap", [(300, 330, 75), (500, 520, 125), (500, 520, 500)])
@pytest.mark.parametrize("kind", list(BLOCKS))
def test_rank_below_the_carried_directions(kind, r, c, cap):
    import torch
    M = need_gpu()
    A = BLOCKS[kind](r, c)
    if kind == "decaying_rows" and (r, cap) == (500, 125):
        # the iterated basis spans thirty decades without any rounding to fill it, more
        # than its Cholesky QR takes: an error, as ever
        with pytest.raises(M.MPOError) as e:
            M.svd_truncated(torch.tensor(A, device="cuda"), cap, "mixed")
        assert e.value.code == -4
        return
    U, X, lam2 = M.svd_truncated(torch.tensor(A, device="cuda"), cap, "mixed")
    U, X = U.cpu().numpy(), X.cpu().numpy()
    s = np.linalg.svd(A, compute_uv=False)
    k = min(cap, int((s > 1e-7 * s[0]).sum()))
    nA = np.linalg.norm(A)
    assert len(lam2) == k
    np.testing.assert_allclose(lam2, s[:k] ** 2, rtol=0, atol=1e-11 * s[0] ** 2)
    assert np.abs(U.conj().T @ U - np.eye(k)).max() < 1e-10
    assert np.linalg.norm(U @ X - U @ (U.conj().T @ A)) <= 1e-7 * nA
    assert np.linalg.norm(A - U @ X) <= np.linalg.norm(s[k:]) + 1e-7 * nA
