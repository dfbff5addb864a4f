"""The normal-equation system on both sides of the condition limit of its
double-float elimination, badly scaled systems included, through the row solve
(spm_selftest_tc_rowpass) against numpy in extended precision.

Bound per element, with scale = max_s |M(i, s)| * sum_s |W(s, c)|: 2^-34 of it
for the operand splitting, R 2^-50 cond of it for the inverse (the bound of an
FP64 factorisation), one FP32 rounding of Z."""
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


@pytest.mark.parametrize("R", [16, 32, 64])
@pytest.mark.parametrize("cond", [1.0, 3.0, 1e2, 1e3, 3e3, 1e4, 1e5, 1e8])
@pytest.mark.parametrize("spread", [0, 30])
def test_inverse_by_the_row_solve(R, cond, spread):
    rng = np.random.default_rng(R + int(cond) + spread)
    Q, _ = np.linalg.qr(rng.standard_normal((R, R)))
    V = (Q * np.logspace(0, np.log10(cond), R)) @ Q.T
    s = 2.0 ** rng.integers(-spread, spread + 1, R)  # exact: the scaled condition stays
    V = 0.5 * (V + V.T) * s[:, None] * s[None, :]
    M = rng.standard_normal((700, R)).astype(np.float32)
    Z, _, _, _ = spm.spm_selftest_tc_rowpass(torch.from_numpy(M).cuda(), torch.from_numpy(V).cuda())
    Vl = (V / s[:, None] / s[None, :]).astype(np.longdouble)
    W = np.linalg.inv(Vl.astype(np.float64)).astype(np.longdouble)
    for _ in range(4):  # refined to extended precision
        W = W + W @ (np.eye(R, dtype=np.longdouble) - Vl @ W)
    W = W / s[:, None] / s[None, :]
    ref = M.astype(np.longdouble) @ W
    scale = np.abs(M).max(1, keepdims=True) * np.abs(W).sum(0, keepdims=True)
    bound = (2.0 ** -34 + cond * R * 2.0 ** -50) * scale + 2.0 ** -23 * np.abs(ref)
    err = np.abs(Z.cpu().numpy().astype(np.longdouble) - ref)
    assert np.all(err <= bound), float((err / bound).max())
