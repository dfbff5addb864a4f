"""Device memory that the library keeps for reuse: given back on request once its
owners are gone, and by a server whose budget it does not fit. Each case in a
process of its own, so that nothing else holds buffers."""
import os
import subprocess
import sys

import pytest

from conftest import ROOT

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

COMMON = """
import torch
import paper_2503_18198_gb300 as spm
ALL = 1 << 62

def tensor(nnz, dims=(4000, 3000, 2000), seed=0):
    g = torch.Generator(device="cuda"); g.manual_seed(seed)
    idx = [torch.randint(0, n, (nnz,), generator=g, device="cuda", dtype=torch.int32) for n in dims]
    return dims, idx, torch.rand(nnz, generator=g, device="cuda")

def factors(dims, R):
    return [torch.randn(n, R, device="cuda") for n in dims]
"""

GIVEN_BACK = COMMON + """
dims, idx, vals = tensor(400_000)
plans = [spm.spmttkrp_plan(dims, idx, vals, 32) for _ in range(3)]
lam = torch.zeros(32, dtype=torch.float64, device="cuda")
fit = torch.zeros(1, dtype=torch.float64, device="cuda")
spm.cpd_als_step(plans[0], factors(dims, 32), lam, fit)
fac = factors(dims, 32)
b = spm.spm_batch_create([plans[1]], [fac], lam, fit)
spm.spm_batch_sweep(b)
torch.cuda.synchronize()
b.destroy()
for p in plans:
    p.destroy()
torch.cuda.synchronize()
kept = spm.spm_memory_trim(ALL)
assert 0 < kept <= 64 << 20, kept
before = torch.cuda.mem_get_info()[0]
assert spm.spm_memory_trim(0) == 0
assert torch.cuda.mem_get_info()[0] - before >= kept
p = spm.spmttkrp_plan(dims, idx, vals, 32)  # and the pool serves again
p.destroy()
"""

SERVER = COMMON + """
dims, idx, vals = tensor(600_000)
need, transient = spm.spmttkrp_plan_bytes_estimate(dims, 600_000, 32, spm.SPM_KAPPA(5))
budget = need + transient + 4 * 32 * sum(dims) + (1 << 20)
assert budget < 64 << 20
S = spm.Server(budget, 8, 0, 131072)
ids = [S.submit(dims, idx, vals, 32, factors(dims, 32), tol=0.0, max_sweeps=2) for _ in range(4)]
for _ in range(40):
    S.step()
    used = S.usage()[0]
    held = spm.spm_memory_trim(ALL)
    # the rest of a block with a live buffer cannot go back
    assert held <= max(budget - used, 32 << 20), (used, held, budget)
    if all(S.info(j).state >= spm.binding.SPM_JOB_DONE for j in ids):
        break
for j in ids:
    assert S.info(j).state == spm.binding.SPM_JOB_DONE
    S.result(j)
S.destroy()
torch.cuda.synchronize()
assert spm.spm_memory_trim(0) == 0
"""


@pytest.mark.parametrize("code", [GIVEN_BACK, SERVER], ids=["given_back", "server"])
def test_memory_kept_for_reuse(code):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    env = dict(os.environ, PYTHONPATH=ROOT)
    res = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=env, capture_output=True,
                         text=True, timeout=300)
    assert res.returncode == 0, res.stderr[-3000:]
