"""The line to four threads per item: the rule on the host, and the results on both sides of it on the GPU."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2402_10914_gb300 import inputs as I

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2402_10914_gb300", "csrc")


def test_rule_counts_what_runs_side_by_side(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "quad_rule_check")
    subprocess.run([nvcc, "-O1", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC,
                    os.path.join(HERE, "quad_rule_check.cu"), "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


# a mesh whose lines (66 x 62: 277 warps) or sides (59 x 58: 432 warps) take four threads per item, and blocks of it
# that do not (6 x 52 = 312 warps of lines; 8 x 60 = 480 warps of sides in the wider blocks)
SIZES = {"lines": (66, 62, 3, 2), "sides": (59, 58, 4, 2)}
CASES = {
    "mixed_bc": lambda nx, ny: I.random_smooth(nx, ny, seed=11, bc=(I.PERIODIC, I.PERIODIC, I.REFLECT, I.OUTFLOW)),
    "smooth_no_limiter": lambda nx, ny: I.random_smooth(nx, ny, seed=12, flux=I.GKS, time_limiter=0),
    "rough_lf": lambda nx, ny: I.random_rough(nx, ny, seed=13, bc=(I.PERIODIC,) * 4, flux=I.LF, time_limiter=0),
    "rough_gks": lambda nx, ny: I.random_rough(nx, ny, seed=15, flux=I.GKS, time_limiter=1),
}


@pytest.mark.gpu
@pytest.mark.parametrize("size", sorted(SIZES))
@pytest.mark.parametrize("name", sorted(CASES))
def test_mesh_below_the_line_equals_its_blocks_above_it(name, size):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    from paper_2402_10914_gb300.solver import DecompSolver, Solver
    __graft_entry__.build()
    nx, ny, px, py = SIZES[size]
    w = CASES[name](nx, ny)
    n = 1 if name.startswith("rough") else 4          # random states lose positivity after a few steps
    with Solver(w.settings) as s:
        s.set_ic(w.W0)
        W0, a0, _, _ = s.get_state()
        assert s.step(n)[0] == n
        W, a, t, _ = s.get_state()
    with DecompSolver(w.settings, px, py) as d:
        d.set_ic(w.W0)
        assert np.array_equal(d.get_state()[1], a0)
        assert d.step(n) == n
        Wd, ad, td, _ = d.get_state()
    assert np.array_equal(W, Wd) and np.array_equal(a, ad) and t == td
