"""A member of a batch whose record-copy waits give up (bounded waits made to
give up at once): it reports the timeout, and no other member's sweep is made
from an spMTTKRP that was left undone -- each either matches its sweep alone bit
for bit or reports the timeout too.  Later sweeps, once the statuses are read
and cleared, are those of the members alone."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2503_18198_gb300 as spm  # noqa: E402

SPM_ERR_TIMEOUT = 6


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    spm.load(build_if_missing=True)


def member(kappa, nnz, R, seed, dtype):
    dims = (700, 500, 300)
    _, idx, vals = synth.coo_random(dims, nnz, seed=seed)
    flags = (spm.SPM_FACTOR_BF16 if dtype == torch.bfloat16 else 0) | spm.SPM_KAPPA(kappa)
    didx = [torch.as_tensor(c, dtype=torch.int32).cuda() for c in idx]
    dval = torch.as_tensor(np.asarray(vals, np.float32)).cuda()
    init = [torch.as_tensor(f).to(dtype).cuda() for f in synth.factors(dims, R, seed=seed)]
    return spm.spmttkrp_plan(dims, didx, dval, R, flags), init


# the failing member has more items than the launch has blocks (every block
# meets it before the others' items), or few; the others are before and after
@pytest.mark.parametrize("kappa,nnz", [(700, 400_000), (2, 60_000)])
@pytest.mark.parametrize("where", [0, 1])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_no_member_is_solved_from_an_unfinished_product(kappa, nnz, where, dtype):
    R = 32
    shapes = [(3, 60_000), (4, 90_000)]
    shapes.insert(where, (kappa, nnz))
    made = [member(k, n, R, 40 + i, dtype) for i, (k, n) in enumerate(shapes)]
    plans = [m[0] for m in made]
    facs = [[f.clone() for f in m[1]] for m in made]
    lam = torch.zeros(R * len(made), dtype=torch.float64, device="cuda")
    fit = torch.zeros(len(made), dtype=torch.float64, device="cuda")
    b = spm.spm_batch_create(plans, facs, lam, fit, 0.0, 8)
    spm.binding.spm_selftest_batch_timeout(b, where)
    status = [spm.spmttkrp_plan_status(p) for p in plans]
    assert status[where] == SPM_ERR_TIMEOUT
    alone = []
    for i, (k, n) in enumerate(shapes):
        plan, init = member(k, n, R, 40 + i, dtype)
        one = [f.clone() for f in init]
        lam1 = torch.zeros(R, dtype=torch.float64, device="cuda")
        spm.cpd_als_step(plan, one, lam1)
        assert spm.spmttkrp_plan_status(plan) == 0
        alone.append((plan, one, lam1))
    for i in range(len(made)):
        if status[i] == 0:
            for a, c in zip(facs[i], alone[i][1]):
                assert torch.equal(a, c), f"member {i} swept from an unfinished product"
        else:
            assert status[i] == SPM_ERR_TIMEOUT
    # the batch restarted from the starting factors is bitwise the members alone
    b.destroy()
    for i, m in enumerate(made):
        for f, f0 in zip(facs[i], m[1]):
            f.copy_(f0)
    b = spm.spm_batch_create(plans, facs, lam, fit, 0.0, 8)
    spm.spm_batch_sweep(b)
    for i, p in enumerate(plans):
        assert spm.spmttkrp_plan_status(p) == 0
        for a, c in zip(facs[i], alone[i][1]):
            assert torch.equal(a, c)
    b.destroy()
