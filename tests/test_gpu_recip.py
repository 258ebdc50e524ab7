"""The panel's reciprocal against the division: the check program is compiled
with the library's flags and run on the GPU."""
import os
import shutil
import subprocess

import pytest

from paper_2102_11910_gb300 import build

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reciprocal_within_one_unit_of_the_division(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "recip_check")
    src = os.path.join(ROOT, "tests", "host", "recip_check.cu")
    inc = ["-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(ROOT, "paper_2102_11910_gb300", "csrc")]
    r = subprocess.run([nvcc, *build.ARCH, *build.NVFLAGS, *inc, src, "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "OK", r.stdout[-2000:]
