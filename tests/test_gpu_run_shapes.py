"""The shapes in which a mode copy is run (blocks and units chosen for its
size, one or several blocks per partition) at their edges, against the FP64
oracle: element-wise within the bound of parity_util, empty rows exactly zero,
repeated runs bitwise equal."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import check_mode_elementwise
from test_gpu_als import gpu_als, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2503_18198_gb300 as spm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# one block per 1024 nonzeros: 1, 2, 32 (last block adds the cut rows) and 33
# blocks (fix-up kernel); kappa kept from 4096 nonzeros per partition on
@pytest.mark.parametrize("nnz,kappa", [(1, 0), (1023, 0), (1025, 0), (32 * 1024, 0),
                                       (32 * 1024 + 1, 0), (5 * 4096, 5), (5 * 4096 - 1, 5),
                                       (150_000, 1), (150_000, 0), (40_000, 5000)])
@pytest.mark.parametrize("R,dtype", [(16, torch.float32), (32, torch.bfloat16),
                                     (24, torch.float32), (100, torch.float32)])
def test_product_in_every_shape(nnz, kappa, R, dtype):
    dims = (1501, 211, 37)  # row runs from a few nonzeros to thousands, empty rows in mode 0
    g = np.random.default_rng(nnz + R)
    idx = [(n * g.random(nnz) ** 2).astype(np.int32) for n in dims]
    vals = g.random(nnz).astype(np.float32)
    Y = [torch.as_tensor(f).to(dtype) for f in synth.factors(dims, R, seed=nnz + R)]
    flags = spm.SPM_FACTOR_BF16 if dtype == torch.bfloat16 else 0
    plan = spm.spmttkrp_plan(dims, [torch.as_tensor(c).cuda() for c in idx],
                             torch.as_tensor(vals).cuda(), R, flags | spm.SPM_KAPPA(kappa))
    fac = [f.cuda() for f in Y]
    for d in range(3):
        out = torch.full((dims[d], R), float("nan"), device="cuda")
        spm.spmttkrp_run(plan, d, fac, out)
        again = torch.full((dims[d], R), float("nan"), device="cuda")
        spm.spmttkrp_run(plan, d, fac, again)
        assert torch.equal(out, again)
        check_mode_elementwise(out.cpu().numpy(), dims, idx, vals, [f.float().numpy() for f in Y], d)


@pytest.mark.parametrize("R,kappa", [(16, 1), (32, 3), (48, 1), (64, 1), (64, 0)])
def test_bf16_sweep_with_shared_partitions(R, kappa):
    """BF16 CP-ALS sums in plan order with 1 to 8 blocks per partition."""
    dims, idx, vals = synth.coo_distinct((900, 300, 60), 60_000, (1.1, None, None), seed=R)
    Y = synth.factors(dims, R, seed=R)
    flags = spm.SPM_FACTOR_BF16 | spm.SPM_KAPPA(kappa)
    plan, fac, lam, fit = gpu_als(dims, idx, vals, Y, 1, flags, torch.bfloat16)
    ofac, olam, ofit = oracle.cpd_als(dims, idx, vals, Y, 1, prec="bf16")
    for d in range(3):
        assert rel(fac[d], ofac[d]) < 2e-3  # one BF16 rounding step apart at most, for few entries
    assert rel(lam, olam) < 1e-3
    assert abs(fit[0] - ofit[0]) < 1e-3
    # the same partitions in one batch: bit for bit the same decomposition
    fac2 = [torch.as_tensor(np.asarray(f, np.float32)).to(torch.bfloat16).cuda() for f in Y]
    if R in (16, 32, 64):
        lam2 = torch.zeros(R, dtype=torch.float64, device="cuda")
        fit2 = torch.zeros(1, dtype=torch.float64, device="cuda")
        b = spm.spm_batch_create([plan], [fac2], lam2, fit2, 0.0, 1)
        spm.spm_batch_sweep(b)
        torch.cuda.synchronize()
        for d in range(3):
            assert np.array_equal(fac2[d].float().cpu().numpy(), fac[d])


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("R", [1, 2, 6, 10, 12, 17, 22, 23, 28, 33, 36, 40, 48, 62, 63, 66, 72, 100,
                               124, 136, 248])
@pytest.mark.parametrize("dims", [(61, 47, 33), (40, 23, 11, 7), (19, 13, 11, 5, 3)])
def test_ranks_between_the_fast_shapes(dims, R, dtype):
    nnz = 3001
    g = np.random.default_rng(R)
    idx = [(n * g.random(nnz) ** 2).astype(np.int32) for n in dims]
    vals = g.random(nnz).astype(np.float32)
    Y = [torch.as_tensor(f).to(dtype) for f in synth.factors(dims, R, seed=R)]
    flags = spm.SPM_FACTOR_BF16 if dtype == torch.bfloat16 else 0
    plan = spm.spmttkrp_plan(dims, [torch.as_tensor(c).cuda() for c in idx],
                             torch.as_tensor(vals).cuda(), R, flags)
    fac = [f.cuda() for f in Y]
    for d in range(len(dims)):
        # guard rows: nothing beyond the output is written
        buf = torch.full((dims[d] + 8, R), 7.0, device="cuda")
        lo = 4 if R % 4 == 0 else 0  # the output starts on a 16-byte boundary
        out = buf[lo:lo + dims[d]]
        spm.spmttkrp_run(plan, d, fac, out)
        assert torch.all(buf[:lo] == 7.0) and torch.all(buf[lo + dims[d]:] == 7.0)
        check_mode_elementwise(out.cpu().numpy(), dims, idx, vals, [f.float().numpy() for f in Y], d)
