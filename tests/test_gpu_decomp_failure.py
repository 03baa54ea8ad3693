"""Which cell a decomposed run names when several blocks lose positivity in the same stage: the first one of the
first failing block, in every run.  (The blocks' updates run side by side.)"""
import numpy as np
import pytest

from paper_2402_10914_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NX, NY = 48, 40


def two_bursts():
    """Streams that recede at Mach 7 in two spots, at a CFL number of 1: positivity is lost at both in the first
    stage, in cells that are below zero by more than one."""
    s = I.Settings(nx=NX, ny=NY, bc=(I.OUTFLOW,) * 4, cfl=1.0, flux=I.GKS)
    rho, u, v, p = np.ones((NY, NX)), np.zeros((NY, NX)), np.zeros((NY, NX)), np.ones((NY, NX))
    for i, j in ((8, 33), (36, 6)):
        u[j - 3:j + 4, i - 3:i], u[j - 3:j + 4, i:i + 3] = -8.0, 8.0
    return s, np.stack([rho, rho * u, rho * v, p / (s.gamma - 1.0) + 0.5 * rho * (u * u + v * v)])


@pytest.mark.parametrize("px,py", [(2, 1), (1, 2), (2, 2), (3, 2), (4, 5)])
def test_the_first_failing_block_names_the_cell(px, py):
    import __graft_entry__
    from paper_2402_10914_gb300 import _lib
    from paper_2402_10914_gb300.solver import DecompSolver, Solver, block_plan
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    s, W0 = two_bursts()
    with Solver(s) as sol:                     # the first stage's state, W + dt/2 L + dt^2/8 dL
        sol.set_ic(W0)
        W, a, _, _ = sol.get_state(device=True)
        u, v = W0[1] / W0[0], W0[2] / W0[0]
        c = np.sqrt(s.gamma * (s.gamma - 1.0) * (W0[3] / W0[0] - 0.5 * (u * u + v * v)))
        dt = s.cfl * min(((s.x1 - s.x0) / NX / (np.abs(u) + c)).min(), ((s.y1 - s.y0) / NY / (np.abs(v) + c)).min())
        L, dL, _, _ = (q.cpu().numpy() for q in sol.residual(W, a, dt))
    W1 = W0 + 0.5 * dt * L + 0.125 * dt * dt * dL
    m = np.minimum(W1[0], W1[0] * W1[3] - 0.5 * (W1[1] ** 2 + W1[2] ** 2))
    assert (np.abs(m) > 1e-3).all() and (m < 0).sum() >= 10
    expected = None
    for b in range(px * py):
        pl = block_plan(s, px, py, b)
        bad = np.argwhere(m[pl["j0"]:pl["j1"], pl["i0"]:pl["i1"]] < 0)
        if len(bad):
            expected = (pl["i0"] + int(bad[0][1]), pl["j0"] + int(bad[0][0]))
            break
    with DecompSolver(s, px, py) as d:
        for _ in range(10):
            d.set_ic(W0)
            with pytest.raises(_lib.DfgksError):
                d.step(3)
            st = d.status()
            assert st["err"] == _lib.ENONPOS and (st["fail_i"], st["fail_j"]) == expected
            W2, a2, t, n = d.get_state()
            assert n == 0 and t == 0.0 and np.array_equal(W2, W0)
