"""The FP32 start of the FP64 form's row Jacobi (32 rows and more) on blocks
with zero rows, equal rows, a rank deficit, repeated singular values and
graded rows, on both sides of its smallest row count, and together with rows
streamed from memory (more than 1024 columns).

The checks and tolerances are those of the sizes without structure."""
import numpy as np
import pytest

from paper_2003_13163_gb300.circuits import random_complex
from tests.gpu_util import need_gpu
from tests.test_gpu_lq_svd import check

pytestmark = pytest.mark.gpu
SIZES = [(20, 50), (33, 1025), (64, 64), (130, 150)]


@pytest.fixture(scope="module")
def M():
    return need_gpu()


@pytest.mark.parametrize("r,c", SIZES)
def test_rank_deficient(M, r, c):
    A = random_complex((r, r // 3), 1) @ random_complex((r // 3, c), 2)
    A[7] = 0
    A[11] = A[3]
    A[0] = 0
    check(M, A, r // 3)


@pytest.mark.parametrize("r,c", SIZES)
def test_zero_and_equal_rows(M, r, c):
    A = random_complex((r, c), 5)
    A[::4] = 0
    for i in range(1, r - 1, 4):
        A[i] = A[i + 1]
    check(M, A, np.linalg.matrix_rank(A))


@pytest.mark.parametrize("r,c", SIZES)
def test_repeated_singular_values(M, r, c):
    s = 2.0 ** -(np.arange(r) // 5)
    U = np.linalg.qr(random_complex((r, r), 3))[0]
    V = np.linalg.qr(random_complex((c, r), 4))[0]
    check(M, (U * s) @ V.conj().T, r)
    check(M, np.eye(r, c, dtype=np.complex128), r)


@pytest.mark.parametrize("r,c", SIZES)
def test_graded_rows(M, r, c):
    check(M, 10.0 ** -np.linspace(0, 9, r)[:, None] * random_complex((r, c), 6), r)


def test_many_rows(M):
    """4096 rows: the FP32 left factor's drift needs the second correction. Rows
    are sigma times orthonormal ones and U orthonormal to the rounding of r
    reflectors and five sweeps of r - 1 rotations on each (both sides of a pair
    change a row): eps sqrt(2 (r + 6 r)), doubled."""
    import torch
    r = 4096
    g = torch.Generator(device="cuda").manual_seed(3)
    A = torch.randn((r, r), dtype=torch.complex128, device="cuda", generator=g)
    U, X, lam2 = M.svd_truncated(A, r, "fp64")
    assert len(lam2) == r
    tol = 2 * 2.2e-16 * np.sqrt(14 * r)
    eye = torch.eye(r, dtype=U.dtype, device="cuda")
    X1 = X / torch.tensor(np.sqrt(lam2), device="cuda")[:, None]
    assert float((X1 @ X1.conj().T - eye).abs().max()) < tol
    assert float((U.conj().T @ U - eye).abs().max()) < tol
    assert float((U @ X - A).abs().max()) < tol * np.sqrt(lam2[0])


def test_no_start_from_a_nan_factor(M):
    """A matrix holding a NaN leaves the FP32 start without a usable factor; the
    solve then runs without it, ends, and the next call is unaffected."""
    import torch
    A = random_complex((64, 70), 1)
    A[3, 3] = np.nan
    M.svd_truncated(torch.tensor(A, device="cuda"), 8, "fp64")
    check(M, random_complex((64, 70), 2), 64)
