"""The integer RAMBO momenta as the device forms them (tests/dir_device_check.cu):
the FP32 estimate behind sin theta for every argument it can get, and the
momenta against the host's, which tests/test_dir.py compares with
high-precision values."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_device_momenta(tmp_path, gpu):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = tmp_path / "dir_device_check"
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-gencode",
                    "arch=compute_103a,code=sm_103a", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_0908_4403_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "dir_device_check.cu"), "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert out[:3] == ["root_estimate", "0", "photon_q"], out
    assert int(out[3]) == 0 and int(out[5]) > 1_000_000, out
