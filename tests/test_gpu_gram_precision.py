"""The Gram of the tensor-core normalisation pass on values whose digits it holds
exactly: the columns' entries lie within a factor of two of each other, so that
24 significant bits fit the digits at R = 16 and 32, and with at most 64 rows the
sums of a digit's products are exact in the FP32 pairs. What is left is the sum
over the digits and its rounding to FP64: 2^-53 of the result and of what a plain
FP64 sum of the digits' parts would add (8 parts, a few 2^-53 of the sum of
magnitudes).  Bound: 2^-51 of sum_i |y_ir y_is|."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2503_18198_gb300 as spm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    spm.load(build_if_missing=True)


@pytest.mark.parametrize("R", [16, 32])
@pytest.mark.parametrize("rows", [1, 8, 40, 64])
@pytest.mark.parametrize("seed", range(4))
def test_gram_of_exact_digits_is_rounded_once(R, rows, seed):
    rng = np.random.default_rng(1000 * R + 10 * rows + seed)
    M = (rng.uniform(1.0, 2.0, (rows, R)) * rng.choice([-1.0, 1.0], (rows, R))).astype(np.float32)
    V = np.eye(R) if seed % 2 else np.eye(R) * 3.0
    _, Y, G, _ = spm.spm_selftest_tc_rowpass(torch.from_numpy(M).cuda(), torch.from_numpy(V).cuda())
    y = Y.cpu().numpy().astype(np.longdouble)
    err = np.abs(G.cpu().numpy().astype(np.longdouble) - y.T @ y)
    bound = 2.0 ** -51 * (np.abs(y).T @ np.abs(y))
    assert np.all(err <= bound), float((err / bound).max())
