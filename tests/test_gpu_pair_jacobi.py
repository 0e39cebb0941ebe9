"""The one-CTA-per-pair row Jacobi SVD (complex128 factorisations) at the
edges of its variants: rows held in registers up to 256 and 1024 columns,
streamed beyond, odd row counts, rank-deficient input and extreme scales.

Tolerances: the solve stops at couplings of 2 eps sqrt(c) ||x_p|| ||x_q||, and
every rotation is unitary to a few eps, so U and U X carry an error of about
eps sqrt(r sweeps) with at most 40 sweeps of r - 1 rotations per row: 10 eps
sqrt(40 r) is asserted, relative to the largest singular value."""
import numpy as np
import pytest

from paper_2003_13163_gb300.circuits import random_complex
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu
EPS = 2.2e-16


@pytest.fixture(scope="module")
def M():
    return need_gpu()


def check(M, X):
    import torch
    r, c = X.shape
    Xt = torch.tensor(X, device="cuda")
    w, Ut = M.svd_rows(Xt, "fp64")
    w, U, Y = w.cpu().numpy(), Ut.cpu().numpy().T, Xt.cpu().numpy()
    ref = np.linalg.svd(X, compute_uv=False)
    tol = 10 * EPS * np.sqrt(40 * r)
    assert np.abs(U.conj().T @ U - np.eye(r)).max() < tol
    assert np.abs(U @ Y - X).max() <= tol * ref[0]
    got = np.sqrt(np.sort(w)[::-1])[:len(ref)]
    assert np.abs(got - ref).max() <= tol * ref[0]
    n = np.linalg.norm(Y, axis=1)
    G = np.abs(Y @ Y.conj().T)
    np.fill_diagonal(G, 0)
    big = n > 1e-12 * n.max()
    assert (G[np.ix_(big, big)] <= 10 * EPS * np.sqrt(max(r, c)) * np.outer(n[big], n[big])).all()


@pytest.mark.parametrize("r,c", [(1, 1), (2, 1), (3, 127), (129, 129), (64, 256), (65, 257), (257, 256), (31, 1024),
                                 (30, 1025), (9, 2100)])
def test_pair_jacobi_sizes(M, r, c):
    check(M, random_complex((r, c), seed=r + c) * np.exp(-np.linspace(0, 9, c))[None, :])


def test_pair_jacobi_rank_deficient(M):
    X = random_complex((20, 6), 1) @ random_complex((6, 50), 2)
    X[7] = 0
    X[11] = X[3]
    check(M, X)


@pytest.mark.parametrize("scale", [1e-75, 1e75])
def test_pair_jacobi_extreme_scales(M, scale):
    """Squared norms of 1e-150 and 1e150: the rotation parameters are formed
    from the couplings' exponents, not from their squares."""
    X = random_complex((24, 40), 5)
    X *= np.exp(-np.linspace(0, 12, 24))[:, None]
    check(M, X * scale)
