"""The normal-equation systems at ranks without a tensor-core solve, on both sides
of the condition limit of their double-float elimination, through a CP-ALS step.

A two-mode tensor with one unit value per row of mode 0 makes the product an exact
copy of rows of factor 1, and factor 1 holds integers (columns scaled by powers of
two), so that its Gram is exact too: what is left of mode 0's update is the
inverse, the row solve and the normalisation. Compared with extended precision.

Bound per element of Z, with scale = max_s |M(i, s)| sum_s |W(s, c)|: R 2^-50 cond
of it for the inverse (as an FP64 factorisation), R 2^-46 for the pairs of the row
solve; then one FP32 rounding of Z, of 1 / lambda and of their product (2^-22 with
what lambda inherits from its column)."""
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


@pytest.mark.parametrize("R", [2, 3, 8, 10, 17, 24, 33, 48, 63])
@pytest.mark.parametrize("cond", [3.0, 1e2, 1e3, 4e3, 1e5])
@pytest.mark.parametrize("spread", [0, 6])
def test_update_of_a_mode_against_extended_precision(R, cond, spread):
    rng = np.random.default_rng(R + int(cond) + spread)
    J = 3 * R + 5
    Q, _ = np.linalg.qr(rng.standard_normal((J, R)))
    P, _ = np.linalg.qr(rng.standard_normal((R, R)))
    Y1 = (Q * np.logspace(0, 0.5 * np.log10(cond), R)) @ P.T
    Y1 = np.rint(Y1 * (1000.0 / np.abs(Y1).max()))
    s = 2.0 ** rng.integers(-spread, spread + 1, R)
    I = 2 * J
    rows = np.arange(I, dtype=np.int32)
    cols = (rows % J).astype(np.int32)
    plan = spm.spmttkrp_plan((I, J), [torch.from_numpy(rows).cuda(), torch.from_numpy(cols).cuda()],
                             torch.ones(I, device="cuda"), R)
    fac = [torch.randn(I, R, device="cuda"), torch.from_numpy((Y1 * s).astype(np.float32)).cuda()]
    lam = torch.zeros(R, dtype=torch.float64, device="cuda")
    spm.cpd_als_step(plan, fac, lam)
    assert spm.spmttkrp_plan_status(plan) == 0

    V = (Y1.T @ Y1).astype(np.longdouble)  # integers below 2^53: exact
    W = np.linalg.inv(V.astype(np.float64)).astype(np.longdouble)
    for _ in range(5):
        W = W + W @ (np.eye(R, dtype=np.longdouble) - V @ W)
    M = Y1[cols].astype(np.longdouble)  # the columns' scales cancel in M W up to one per column
    Z = M @ W
    norm = np.sqrt((Z * Z).sum(0))
    d = np.sqrt(np.diag(V).astype(np.float64))
    unit = V.astype(np.float64) / d[:, None] / d[None, :]
    scale = np.abs(M).max(1, keepdims=True) * np.abs(W).sum(0, keepdims=True)
    eps = R * 2.0 ** -50 * np.linalg.cond(unit) + R * 2.0 ** -46
    dz = eps * scale / norm
    ref = Z / norm
    bound = dz + np.abs(ref) * (2.0 ** -22 + np.sqrt((dz * dz).sum(0)))
    err = np.abs(fac[0].cpu().numpy().astype(np.longdouble) - ref)
    assert np.all(err <= bound), float((err / bound).max())
