"""Memory that is handed back while another device is current: the wait before
it has to be for the device that the memory lies on.  Shown on the host, on a
fake runtime (a wait on the wrong device would be a race on real memory)."""
import glob
import os
import re
import shutil
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2503_18198_gb300", "csrc")

PROBE = r"""
#include <cstdio>
#include "device_drain.h"
struct Fake {
  int current, fail_set, synced = -1, order = 0;
  bool get(int* d) { *d = current; return true; }
  bool set(int d) { if (fail_set) return false; current = d; return true; }
  bool sync() { synced = current; ++order; return true; }
};
int main() {
  Fake same{2, 0}, other{0, 0}, broken{0, 1};
  if (!spm::drain_device(same, 2) || same.synced != 2 || same.current != 2) return 1;
  if (!spm::drain_device(other, 3) || other.synced != 3 || other.current != 0) return 2;
  if (spm::drain_device(broken, 3) || broken.synced != -1 || broken.current != 0) return 3;
  return 0;
}
"""


def test_drain_waits_for_the_named_device_and_restores_the_current_one(tmp_path):
    cxx = shutil.which("g++") or pytest.skip("no host compiler")
    (tmp_path / "probe.cpp").write_text(PROBE)
    exe = str(tmp_path / "probe")
    subprocess.run([cxx, "-std=c++17", "-I" + CSRC, str(tmp_path / "probe.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0


def test_no_owner_waits_for_whatever_device_is_current():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        if os.path.basename(path) == "dev_alloc.cu":
            continue
        code = re.sub(r"//[^\n]*", "", open(path).read())
        assert "cudaDeviceSynchronize" not in code, path
