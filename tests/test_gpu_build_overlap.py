"""A plan build does not wait for work of other streams: a server builds the
plans of queued jobs while a sweep runs."""
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


# sort scratch below and above the size that the buffer pool serves
@pytest.mark.parametrize("nnz", [100_000, 1_500_000, 6_000_000])
@pytest.mark.parametrize("flags", [0, spm.SPM_FACTOR_BF16])
def test_build_ends_while_another_stream_is_busy(nnz, flags):
    dims = (60_000, 50_000, 40_000)
    g = torch.Generator(device="cuda")
    g.manual_seed(nnz)
    idx = [torch.randint(0, n, (nnz,), generator=g, device="cuda", dtype=torch.int32) for n in dims]
    vals = torch.rand(nnz, generator=g, device="cuda")
    build, busy = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(2):  # kernels loaded, clocks up
        spm.spmttkrp_plan(dims, idx, vals, 32, flags, build).destroy()
    done = torch.cuda.Event()
    with torch.cuda.stream(busy):
        torch.cuda._sleep(1_500_000_000)  # about 0.75 s; a build takes milliseconds
        done.record()
    plan = spm.spmttkrp_plan(dims, idx, vals, 32, flags, build)
    ended_first = not done.query()
    torch.cuda.synchronize()
    plan.destroy()
    assert ended_first, "the build waited for the other stream's work"


def test_large_scratch_is_given_back_when_the_build_returns():
    """6M nonzeros: 144 MB of sort scratch, which no plan may go on holding.
    Slack: the buffer pool's 64 MB and the driver's granules."""
    dims, nnz = (60_000, 50_000, 40_000), 6_000_000
    idx = [torch.randint(0, n, (nnz,), device="cuda", dtype=torch.int32) for n in dims]
    vals = torch.rand(nnz, device="cuda")
    spm.spmttkrp_plan(dims, idx, vals, 32).destroy()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    plans = [spm.spmttkrp_plan(dims, idx, vals, 32) for _ in range(4)]
    torch.cuda.synchronize()
    taken = before - torch.cuda.mem_get_info()[0]
    assert taken < sum(spm.spmttkrp_plan_bytes(p) for p in plans) + (100 << 20)
    for p in plans:
        p.destroy()
