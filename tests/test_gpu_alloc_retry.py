"""A CP-ALS step that ran out of memory while it made its workspace can be tried
again: it goes on from what was allocated, so the plan ends up holding the bytes
of one that never failed."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2503_18198_gb300 as spm  # noqa: E402

SPM_ERR_OOM = 3


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    spm.load(build_if_missing=True)
    yield
    spm.binding.spm_inject_alloc_failure(-1)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("R", [24, 32])
def test_step_tried_again_after_a_failed_allocation(dtype, R):
    dims, idx, vals = synth.coo_distinct((900, 300, 60), 60_000, (1.1, None, None), seed=9)
    flags = (spm.SPM_FACTOR_BF16 if dtype == torch.bfloat16 else 0) | spm.SPM_KAPPA(3)
    didx = [torch.as_tensor(c).cuda() for c in idx]
    dval = torch.as_tensor(vals).cuda()
    init = [torch.as_tensor(f).to(dtype).cuda() for f in synth.factors(dims, R, seed=9)]

    def run(k):
        """(allocations failed, plan bytes, results) with the k-th allocation of the step failing."""
        plan = spm.spmttkrp_plan(dims, didx, dval, R, flags)
        fac = [f.clone() for f in init]
        lam = torch.zeros(R, dtype=torch.float64, device="cuda")
        failed = 0
        spm.binding.spm_inject_alloc_failure(k)
        try:
            spm.cpd_als_step(plan, fac, lam)
        except spm.SpmError as e:
            assert e.status == SPM_ERR_OOM
            failed = 1
        spm.binding.spm_inject_alloc_failure(-1)
        if failed:
            spm.cpd_als_step(plan, fac, lam)
        assert spm.spmttkrp_plan_status(plan) == 0
        out = failed, spm.spmttkrp_plan_bytes(plan), fac + [lam]
        plan.destroy()
        return out

    _, want_bytes, want = run(-1)
    for k in range(20):
        failed, held, got = run(k)
        if not failed:
            break
        assert held == want_bytes, f"allocation {k}"
        for a, b in zip(got, want):
            assert torch.equal(a, b)
    # every rank has nine buffers; the digit tile and the shared partitions' three come on top
    assert k == 9 + (R == 32) + 3 * (dtype == torch.bfloat16)
