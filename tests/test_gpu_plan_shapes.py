"""Mode copies, partitions and work units at the edges of the build kernels'
tiles and digits, bit-exact against the oracle's permutation and formulas:
tiles of 2048 and 8192 pairs, segments of 512 positions, one- and two-digit
coordinates, keys of one and of two words, many and few nonzeros per unit."""
import numpy as np
import pytest

from test_gpu_mttkrp import check_copies

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2503_18198_gb300 as spm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def build(dims, nnz, kappa, R=32, skew=2, flags=0):
    g = np.random.default_rng(nnz + len(dims))
    idx = [(n * g.random(nnz) ** skew).astype(np.int64).astype(np.int32) for n in dims]
    plan = spm.spmttkrp_plan(dims, [torch.as_tensor(c).cuda() for c in idx],
                             torch.as_tensor(g.random(nnz).astype(np.float32)).cuda(), R,
                             flags | spm.SPM_KAPPA(kappa))
    return plan, idx


@pytest.mark.parametrize("nnz", [1, 31, 511, 512, 513, 1024, 2047, 2048, 2049, 4096 + 7, 100_003])
@pytest.mark.parametrize("kappa", [1, 7, 0])
def test_sizes_around_tiles_and_segments(nnz, kappa):
    plan, idx = build((1025, 1024, 3), nnz, kappa)
    check_copies(plan, idx, kappa or None)


@pytest.mark.parametrize("dims", [(1, 1, 1), (1, 5, 1), (2, 1 << 20, (1 << 20) + 1),
                                  ((1 << 30) + 7, 1025, 2), ((1 << 24), (1 << 24), (1 << 24)),
                                  (1 << 17, 1 << 17, 1 << 17, 1 << 17), (3, 1, 4, 1, 5, 9, 2)])
def test_digits_and_key_words(dims):
    plan, idx = build(dims, 5003, 5)
    check_copies(plan, idx, 5)


def test_large_tiles_and_units_by_search():
    plan, idx = build((4000, 70_000, 301), (1 << 20) + 8192 + 5, 16, R=64, skew=3)
    check_copies(plan, idx, 16)
    spm.spmttkrp_plan_repartition(plan, 5)
    check_copies(plan, idx, 5)
