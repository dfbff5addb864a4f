"""The partition autotuner times launches that differ and picks among them; the
run that it leaves, and a plan built with that count, agree bit for bit."""
import numpy as np
import pytest

import synth
from parity_util import check_mode_elementwise

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2503_18198_gb300 as spm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    spm.load(build_if_missing=True)


def make(nnz, dtype, kappa, R=32):
    g = np.random.default_rng(nnz)
    dims = (9001, 1511, 307)
    idx = [(n * g.random(nnz) ** 2).astype(np.int32) for n in dims]
    vals = g.random(nnz).astype(np.float32)
    flags = (spm.SPM_FACTOR_BF16 if dtype == torch.bfloat16 else 0) | spm.SPM_KAPPA(kappa)
    Y = [torch.as_tensor(f).to(dtype).cuda() for f in synth.factors(dims, R, seed=7)]

    def plan(k):
        return spm.spmttkrp_plan(dims, [torch.as_tensor(c).cuda() for c in idx],
                                 torch.as_tensor(vals).cuda(), R,
                                 (flags & ~(0xFFFF << 16)) | spm.SPM_KAPPA(k))
    return dims, idx, vals, Y, plan


@pytest.mark.parametrize("had", [0, 5])
def test_equal_launches_share_a_time_and_keep_the_plans_count(had):
    sms = spm.spm_device_sm_count()
    _, _, _, Y, plan = make(20_000, torch.float32, had)
    p = plan(had)
    had = had or 2 * sms
    chosen, ms = spm.spmttkrp_plan_autotune(p, Y, [sms, 2 * sms, 5, 3 * sms], reps=2)
    assert len(set(ms)) == 1  # 20 blocks each: one launch
    assert chosen == had


def test_a_whole_number_of_partitions_per_sm_is_its_own_launch():
    sms = spm.spm_device_sm_count()
    dims, idx, vals, Y, plan = make(4096 * 2 * sms, torch.float32, 0)
    p = plan(0)
    ks = [sms, 2 * sms, sms - 1]
    chosen, ms = spm.spmttkrp_plan_autotune(p, Y, ks, reps=2)
    assert ms[1] == ms[2]  # sms - 1 is cut for the device: 2 blocks per SM
    assert chosen in ks and ms[ks.index(chosen)] == min(ms)
    for k in (sms, 2 * sms):  # the runs themselves, against the oracle and a fresh plan
        spm.spmttkrp_plan_repartition(p, k)
        fresh = plan(k)
        for d in range(3):
            a = torch.full((dims[d], 32), float("nan"), device="cuda")
            b = torch.full((dims[d], 32), float("nan"), device="cuda")
            spm.spmttkrp_run(p, d, Y, a)
            spm.spmttkrp_run(fresh, d, Y, b)
            assert torch.equal(a, b)
            check_mode_elementwise(a.cpu().numpy(), dims, idx, vals, [f.cpu().numpy() for f in Y], d)


def test_bf16_candidates_are_timed_as_a_sweep_runs_them():
    """A BF16 sweep shares a partition between blocks by the plan's units, so every
    count is a launch of its own there, while a product cuts all of these alike."""
    ks = [16, 40, 100, 304]
    for dtype, distinct in ((torch.float32, False), (torch.bfloat16, True)):
        _, _, _, Y, plan = make(150_000, dtype, 0)
        p = plan(0)
        chosen, ms = spm.spmttkrp_plan_autotune(p, Y, ks, reps=2)
        assert (len(set(ms)) > 1) == distinct
        assert ms[ks.index(chosen)] == min(ms)
        lam = torch.zeros(32, dtype=torch.float64, device="cuda")
        got = [y.clone() for y in Y]
        spm.cpd_als_step(p, got, lam)
        want = [y.clone() for y in Y]
        spm.cpd_als_step(plan(chosen), want, lam)
        for a, b in zip(got, want):
            assert torch.equal(a, b)
