"""Memory-lean plans at ranks between the fast shapes: products and sweeps are
bitwise those of the full plan there too (the kernels of both take the same
lanes and chunks)."""
import pytest

import oracle  # noqa: F401
import synth
from test_gpu_lean import bits, build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2503_18198_gb300 as spm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    spm.load(build_if_missing=True)


CASES = [
    ((300, 200, 100), 20_000, (1.2, 1.2, 1.2)),
    ((64, 48, 32, 6), 5_000, (None, None, None, None)),
    ((400, 90, 2, 30, 11), 30_000, (1.1, 1.1, None, None, None)),
    ((500, 70), 4_000, (1.1, None)),
]


# one rank of every masked shape of either type, and ranks that keep the scalar one
@pytest.mark.parametrize("R", [5, 10, 12, 22, 24, 36, 40, 48, 63, 66, 100, 136, 192])
@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("dtype,fflag", [(torch.float32, spm.SPM_FACTOR_FP32),
                                         (torch.bfloat16, spm.SPM_FACTOR_BF16)])
def test_lean_plan_equals_full_plan_bitwise_between_the_fast_ranks(R, case, dtype, fflag):
    dims, nnz, alphas = CASES[case]
    dims, _, _, full = build(dims, nnz, R, alphas, 90 + R, fflag)
    _, _, _, lean = build(dims, nnz, R, alphas, 90 + R, fflag | spm.SPM_PLAN_LEAN)
    Y = [torch.as_tensor(f).to(dtype).cuda().contiguous() for f in synth.factors(dims, R, seed=R)]
    for d in range(len(dims)):
        a = torch.full((dims[d], R), float("nan"), device="cuda")
        b = torch.full((dims[d], R), float("nan"), device="cuda")
        spm.spmttkrp_run(full, d, Y, a)
        spm.spmttkrp_run(lean, d, Y, b)
        assert torch.equal(a, b), f"mode {d}"
    if R <= 64:
        got = []
        for plan in (full, lean):
            fac = [y.clone() for y in Y]
            lam = torch.zeros(R, dtype=torch.float64, device="cuda")
            spm.cpd_als_step(plan, fac, lam)
            got.append((spm.spmttkrp_plan_status(plan), lam, fac))
        assert got[0][0] == got[1][0]
        if got[0][0] == 0:
            assert torch.equal(got[0][1], got[1][1])
            for x, y in zip(got[0][2], got[1][2]):
                assert torch.equal(bits(x), bits(y))
