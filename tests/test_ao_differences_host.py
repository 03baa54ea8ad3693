"""WENO-AO in undivided differences against its sub-stencil polynomials in long double, on the host: data from far below
the smoothness epsilon to magnitudes where the scaled weights overflow and the ratios are used instead."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2402_10914_gb300", "csrc")


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("ao") / "ao_differences_check")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC,
                    os.path.join(HERE, "ao_differences_check.cu"), "-o", out], check=True, capture_output=True)
    return out


@pytest.mark.parametrize("exponent", [-12, -4, -2, 0, 2, 8, 9.5, 14, 30])
def test_difference_form_is_the_same_reconstruction(exe, exponent):
    r = subprocess.run([exe, str(exponent)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
