"""The launches that a plan states for a product are those that are made (as the
profiler sees them)."""
import numpy as np
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
    profiled(lambda: torch.ones(8, device="cuda") + 1)  # the first session sees no events
    if not profiled(lambda: torch.ones(8, device="cuda") + 1):
        pytest.skip("the profiler sees no kernels here")


def profiled(call):
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CPU,
                                            torch.profiler.ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    return [e.name for e in prof.events() if e.device_type == torch.autograd.DeviceType.CUDA]


# 20 blocks (no fix-up of its own), few partitions cut into more than 32 blocks,
# many blocks, one partition per SM, Scheme 1, fibre copies with empty rows
@pytest.mark.parametrize("nnz,kappa,flags,blocks", [
    (20_000, 0, 0, 20), (32 * 1024, 2, 0, 32), (200_000, 8, 0, 128), (200_000, 0, 0, 196),
    (20_000, 5, spm.SPM_POLICY_SCHEME1, 5), (20_000, 7, spm.SPM_POLICY_SCHEME2, 20),
    (20_000, 7, spm.SPM_PLAN_FIBRE, 7), (20_000, 1, spm.SPM_PLAN_FIBRE, 1), (0, 0, 0, 0)])
def test_stated_launches_are_those_made(nnz, kappa, flags, blocks):
    dims = (1501, 211, 37)
    g = np.random.default_rng(nnz)
    idx = [(n * g.random(nnz) ** 2).astype(np.int32) for n in dims]
    plan = spm.spmttkrp_plan(dims, [torch.as_tensor(c).cuda() for c in idx],
                             torch.as_tensor(g.random(nnz).astype(np.float32)).cuda(), 32,
                             flags | spm.SPM_KAPPA(kappa))
    Y = [torch.as_tensor(f).cuda() for f in synth.factors(dims, 32, seed=1)]
    for d in range(3):
        out = torch.empty(dims[d], 32, device="cuda")
        spm.spmttkrp_run(plan, d, Y, out)
        torch.cuda.synchronize()
        names = profiled(lambda: spm.spmttkrp_run(plan, d, Y, out))
        made = [n for n in names if "kernel" in n]
        kernels, nblocks = spm.spmttkrp_plan_launches(plan, d)
        assert kernels == len(made), names
        assert nblocks == blocks
