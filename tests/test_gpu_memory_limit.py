"""A memory limit with no room for the optional workspaces (the FP64 form's LQ
step, the K parts of the split product) leaves the handle on the routes that
need none; the entropies agree with the unlimited handle's.

Tolerance: both routes factor to FP64 rounding (the precision form to 2^-42),
far below the 1e-9 asserted on the entropies of an untruncated circuit."""
import re

import numpy as np
import pytest

from paper_2003_13163_gb300.circuits import random_circuit
from tests.gpu_util import need_gpu, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    return need_gpu()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_tight_memory_limit(M, precision):
    c = random_circuit(8, 4, 0.02, seed=3)
    with pytest.raises(M.MPOError) as e:
        M.MPO(8, 256, precision, arena_cap_bytes=1)
    need = int(re.search(r"needed \((\d+) B\)", str(e.value)).group(1))
    S, tr, _, m = run_gpu(M, c, 256, precision)
    Sl, trl, _, ml = run_gpu(M, c, 256, precision, arena_cap_bytes=need)
    assert ml.device_bytes() < m.device_bytes()
    assert np.abs(S - Sl).max() < 1e-9
    np.testing.assert_allclose(trl, tr, atol=1e-7 if precision == "mixed" else 1e-12)
    m.close()
    ml.close()
