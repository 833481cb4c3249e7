"""Events whose photons are parallel to rounding (mass squared at or below 0,
once in 1e16) have no momenta to speak of and pass no cuts, in FP32 or FP64
(tests/cuts_check.cu): a normal event passes, the others do not."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_momenta_that_are_no_numbers_pass_no_cuts(tmp_path, gpu):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = tmp_path / "cuts_check"
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_0908_4403_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "cuts_check.cu"), "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split("\n")[:-1]
    assert len(out) == 12
    for k, line in enumerate(out):
        assert line == ("1 1" if k % 6 == 0 else "0 0"), (k, out)
