"""The reverse sweep's building blocks as the kernels use them, on the host: face basis and projections of
differences against central differences, and the taped sweeps inside tapes of exactly the library's size."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2402_10914_gb300", "csrc")


@pytest.mark.parametrize("name,lines", [("difference_reverse_check", 2), ("tape_bounds_check", 8)])
def test_host_check(tmp_path, name, lines):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / name)
    subprocess.run([nvcc, "-O1", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC,
                    os.path.join(HERE, name + ".cu"), "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.count(" ok") == lines, r.stdout
