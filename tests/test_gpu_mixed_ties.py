"""The precision form on blocks with exactly equal singular values, exactly zero
rows or a rank deficit, as structured gates and unsaturated bonds give them:
nothing there separates the FP32 vectors, and the first-order correction meets
pairs whose values and coupling are both exactly zero apart.

Tolerances are the form's: U from FP64-accurate products ends orthonormal to
1e-10, the kept block is U U^H A and misses no more of A than the best one, each
to 1e-7 of |A|; the squared values agree to 1e-11 of the largest."""
import numpy as np
import pytest

from paper_2003_13163_gb300.circuits import layer_bonds, random_complex
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    return need_gpu()


def unitary(r, seed):
    return np.linalg.qr(random_complex((r, r), seed))[0]


BLOCKS = {
    "identity": lambda r: np.eye(r, dtype=np.complex128),
    "half_rows_zero": lambda r: np.where(np.arange(r)[:, None] % 2 == 0, random_complex((r, r + 3), r), 0.0),
    "flat": lambda r: 0.5 * unitary(r, r),
    "repeated_diagonal": lambda r: np.diag(2.0 ** -(np.arange(r) // 4).astype(float)).astype(np.complex128),
    "equal_rows": lambda r: np.repeat(random_complex((r // 2, r + 1), r), 2, axis=0),
    "rank_deficient": lambda r: random_complex((r, r // 4), 1) @ random_complex((r // 4, r + 5), 2),
}


@pytest.mark.parametrize("r", [32, 48, 64, 130])
@pytest.mark.parametrize("truncate", [False, True])
@pytest.mark.parametrize("kind", list(BLOCKS))
def test_ties(M, kind, truncate, r):
    import torch
    A = BLOCKS[kind](r)
    cap = r // 4 if truncate else r
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


def test_cnot_circuit_matches_fp64_form(M):
    """Noisy CNOTs from the product state keep the state a mixture of basis
    states: theta' has zero rows and equal values. |dS| <= 1e-6 is the form's bar."""
    n, chi = 12, 64
    cnot = np.eye(4)[[0, 1, 3, 2]].astype(np.complex128)
    S = {}
    for precision in ("fp64", "mixed"):
        with M.MPO(n, chi, precision) as m:
            S[precision] = []
            for t in range(8):
                m.apply_layer(t % 2, np.array([cnot] * len(layer_bonds(n, t % 2))), 0.05)
                s, trace, _ = m.entropy()
                assert abs(trace - 1.0) < 1e-6
                S[precision].append(s)
    assert np.abs(np.array(S["fp64"]) - np.array(S["mixed"])).max() <= 1e-6
