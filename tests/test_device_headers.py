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
