"""Fibre plans hold no workspace that their kernels never read: with BF16
factors the plan's own bytes are those with FP32 factors (the layout, the
MTTKRP and the CP-ALS workspace do not depend on the factor type)."""
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


@pytest.mark.parametrize("kappa", [0, 2])
def test_fibre_plan_bytes_do_not_depend_on_the_factor_type(kappa):
    dims, idx, vals = synth.coo_distinct((900, 300, 60), 60_000, (1.1, None, None), seed=5)
    held = []
    for flags, dtype in ((0, torch.float32), (spm.SPM_FACTOR_BF16, torch.bfloat16)):
        plan = spm.spmttkrp_plan(dims, [torch.as_tensor(c).cuda() for c in idx],
                                 torch.as_tensor(vals).cuda(), 32,
                                 flags | spm.SPM_PLAN_FIBRE | spm.SPM_KAPPA(kappa))
        fac = [torch.as_tensor(f).to(dtype).cuda() for f in synth.factors(dims, 32, seed=5)]
        spm.cpd_als_step(plan, fac, torch.zeros(32, dtype=torch.float64, device="cuda"))
        assert spm.spmttkrp_plan_status(plan) == 0
        held.append(spm.spmttkrp_plan_bytes(plan))
        plan.destroy()
    assert held[0] == held[1]
