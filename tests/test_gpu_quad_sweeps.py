"""The sweeps with four threads per face line and side (small meshes) against those with one: a mesh above the
line between them, whole and in blocks below it, bit for bit."""
import numpy as np
import pytest

from paper_2402_10914_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = {
    "mixed_bc": lambda: I.random_smooth(130, 121, seed=11, bc=(I.PERIODIC, I.PERIODIC, I.REFLECT, I.OUTFLOW)),
    "smooth_no_limiter": lambda: I.random_smooth(129, 122, seed=12, flux=I.GKS, time_limiter=0),
    "rough_lf": lambda: I.random_rough(131, 120, seed=13, bc=(I.PERIODIC,) * 4, flux=I.LF, time_limiter=0),
    "blast_walls": lambda: I.blast(126),
    "quadrants": lambda: I.quadrants(125, seed=4),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_blocks_below_the_line_equal_the_mesh_above_it(name):
    import __graft_entry__
    from paper_2402_10914_gb300.solver import DecompSolver, Solver
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    w = CASES[name]()
    n = 1 if name.startswith("rough") else 4          # random states lose positivity after a few steps
    with Solver(w.settings) as s:
        s.set_ic(w.W0)
        assert s.step(n)[0] == n
        W, a, t, _ = s.get_state()
        cnt = s.counters()
    with DecompSolver(w.settings, 3, 3) as d:
        d.set_ic(w.W0)
        assert d.step(n) == n
        Wd, ad, td, _ = d.get_state()
        st = d.status()
    assert np.array_equal(W, Wd) and np.array_equal(a, ad) and t == td
    # blocks repeat the lines and faces of their shared boundaries, so their counters are never below
    for key in ("df_normal", "df_tangential", "fallbacks"):
        assert st[key] >= cnt[key], key
