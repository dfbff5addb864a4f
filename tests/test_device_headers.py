"""Compile-time properties of the device headers that a run cannot show safely
or that depend on a build switch, through the compiler's front end (no GPU)."""
import os
import subprocess

import pytest

from paper_2503_18198_gb300 import _build


@pytest.fixture(scope="module")
def nvcc():
    try:
        return _build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")


def check(nvcc, tmp_path, body, *flags):
    src = tmp_path / "probe.cu"
    src.write_text('#include "batch_kernels.cuh"\nnamespace spm {\n' + body + "\n}\n")
    res = subprocess.run([nvcc, *_build.ARCH, *_build.NVCC_FLAGS, *flags, "-I" + _build.CSRC,
                          "-cuda", str(src), "-o", str(tmp_path / "probe.ii")],
                         capture_output=True, text=True)
    assert res.returncode == 0, res.stderr


def test_staged_gram_rows_take_16_byte_loads(nvcc, tmp_path):
    """The CUDA-core Gram reads its staged rows as float4: the shared struct and
    the row stride have to be multiples of 16 bytes."""
    check(nvcc, tmp_path, "\n".join(
        f"static_assert(alignof(GramSmem<{g}>) % 16 == 0 && GramShape<{g}>::LD % 4 == 0, \"\");"
        for g in (1, 2, 4)))


def test_partitions_asked_for_per_sm_are_what_a_run_takes(nvcc, tmp_path):
    """One and two partitions per SM are different launches from 4096 nonzeros
    per partition on (one block each), so that the autotuner's default
    candidates are a choice; below, and at counts that leave SMs idle, the copy
    is cut for the device."""
    kx = "mttkrp_shape(0, {nnz}LL, {kappa}, 128, {sms}).kx"
    cases = []
    for sms in (148, 152):
        for per in (1, 2, 3):
            k = per * sms
            cases += [(4096 * k, k, sms, k), (50_000_000, k, sms, k), (4096 * k - 1, k, sms, 2 * sms)]
        cases += [(50_000_000, sms - 1, sms, 2 * sms), (50_000_000, 1, sms, 16), (50_000_000, 3, sms, 48),
                  (50_000_000, sms + 1, sms, 2 * sms), (50_000_000, 2 * sms + 1, sms, 2 * sms + 1),
                  (1, 1, sms, 1), (20_000, sms, sms, 20), (20_000, 2 * sms, sms, 20), (33_000, 2, sms, 32),
                  (33_000, 3, sms, 33)]
    check(nvcc, tmp_path, "\n".join(
        f"static_assert({kx.format(nnz=n, kappa=k, sms=s)} == {want}, \"{n} {k} {s}\");"
        for n, k, s, want in cases))


@pytest.mark.parametrize("tc", [1, 0])
def test_the_digit_tile_exists_for_the_ranks_of_the_tensor_core_solve_only(nvcc, tmp_path, tc):
    """The system kernel writes either the digit tile or V^-1 itself: a tile held
    for a rank whose solve is on the CUDA cores would leave that solve nothing."""
    check(nvcc, tmp_path, "\n".join(
        f"static_assert((als_wdig_bytes({r}) != 0) == tc_solve_rank({r}), \"rank {r}\");"
        for r in (8, 16, 24, 32, 64)), f"-DSPM_ALS_TC={tc}")
