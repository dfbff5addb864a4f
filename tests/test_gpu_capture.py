"""A CP-ALS step captured in a CUDA graph after the plan was repartitioned: the
captured sweep is bitwise the one launched directly."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2503_18198_gb300 as spm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    spm.load(build_if_missing=True)


# partition counts before and at the capture: the BF16 sweep shares a partition
# between blocks at few of them and needs buffers that grow with the count
@pytest.mark.parametrize("first,then", [(0, 2), (2, 5), (5, 2), (2, 0)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_step_captured_after_a_repartition(first, then, dtype):
    R = 32
    dims, idx, vals = synth.coo_distinct((900, 300, 60), 120_000, (1.1, None, None), seed=3)
    flags = spm.SPM_FACTOR_BF16 if dtype == torch.bfloat16 else 0
    didx = [torch.as_tensor(c).cuda() for c in idx]
    dval = torch.as_tensor(vals).cuda()
    init = [torch.as_tensor(f).to(dtype).cuda() for f in synth.factors(dims, R, seed=3)]

    def run(captured):
        plan = spm.spmttkrp_plan(dims, didx, dval, R, flags | spm.SPM_KAPPA(first))
        fac = [f.clone() for f in init]
        lam = torch.zeros(R, dtype=torch.float64, device="cuda")
        fit = torch.zeros(1, dtype=torch.float64, device="cuda")
        spm.cpd_als_step(plan, fac, lam, fit)
        spm.spmttkrp_plan_repartition(plan, then)
        torch.cuda.synchronize()
        if captured:
            g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
            s.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(s):
                with torch.cuda.graph(g, stream=s):
                    spm.cpd_als_step(plan, fac, lam, fit)
            torch.cuda.current_stream().wait_stream(s)
            g.replay()
        else:
            spm.cpd_als_step(plan, fac, lam, fit)
        assert spm.spmttkrp_plan_status(plan) == 0
        return fac + [lam, fit]

    for a, b in zip(run(True), run(False)):
        assert torch.equal(a, b)
