"""CP-ALS at ranks on both sides of every block-shape limit of the update
kernels, against the FP64 oracle.

Bounds as in test_gpu_als.py: factors and weights after one sweep within 1e-4
(FP32 MTTKRP and storage, FP64 system), fit within 1e-3."""
import numpy as np
import pytest

import oracle
import synth
from test_gpu_als import gpu_als, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("R", [1, 2, 15, 17, 31, 32, 33, 47, 63, 64])
def test_one_sweep_at_rank_edges(R):
    dims, idx, vals = synth.coo_distinct((611, 403, 259), 30000, (1.1, None, None), seed=70 + R)
    Y = synth.factors(dims, R, seed=70 + R)
    _, fac, lam, fit = gpu_als(dims, idx, vals, Y, 1)
    ofac, olam, ofit = oracle.cpd_als(dims, idx, vals, Y, 1, prec="fp32")
    for d in range(3):
        assert rel(fac[d], ofac[d]) < 1e-4
    assert rel(lam, olam) < 1e-4
    assert abs(fit[0] - ofit[0]) < 1e-3
