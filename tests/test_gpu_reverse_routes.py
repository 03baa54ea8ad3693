"""The reverse of a stage by every route the reverse's memory can lead to: both directions at once or one after the
other, with all tapes, the ratios' alone or none.  Each against the oracle, at odd and degenerate sizes, and by
which route the handle's bytes show it went."""
import numpy as np
import pytest

import oracle
from paper_2402_10914_gb300 import inputs as I
from tests.parity_util import comp_rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def sizes(s):
    """Bytes of a direction's adjoints (27 values a line, 25 a face side), of its ratio tapes and of its GKS tapes."""
    up4 = lambda n: (n + 3) // 4 * 4  # noqa: E731
    lines = up4(max((s.nx + 1) * (s.ny + 4), (s.ny + 1) * (s.nx + 4)))
    sides = up4(2 * max((s.nx + 1) * s.ny, (s.ny + 1) * s.nx))
    return 8 * (27 * lines + 25 * sides), 8 * (48 * lines + 24 * sides), 8 * 39 * sides


CASES = {
    "gks_rough": (lambda: I.random_rough(23, 17, seed=51, flux=I.GKS, time_limiter=1), True),
    "gks_reflect": (lambda: I.random_smooth(19, 26, seed=52, bc=(I.REFLECT,) * 4, flux=I.GKS, time_limiter=1), False),
    "gks_tau_n": (lambda: I.random_smooth(14, 11, seed=53, flux=I.GKS, time_limiter=0, tau_reading=1), False),
    "gks_one_column": (lambda: I.random_rough(1, 9, seed=54, flux=I.GKS, time_limiter=1), True),
    "lf_periodic": (lambda: I.random_rough(21, 16, seed=55, bc=(I.PERIODIC,) * 4, flux=I.LF, time_limiter=0), True),
    "lf_limiter": (lambda: I.random_rough(16, 33, seed=56, flux=I.LF, time_limiter=1), True),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_routes_agree_with_the_oracle(name):
    from paper_2402_10914_gb300.solver import Solver, adjoint_residual
    make, scattered = CASES[name]
    w = make()
    s = w.settings
    rng = np.random.default_rng(9)
    alpha = rng.uniform(0.0, 1.0, (s.ny, s.nx)) if scattered else np.ones((s.ny, s.nx))
    dt = 0.4 * oracle.cfl_dt(s, w.W0)
    bars = [rng.normal(size=w.W0.shape) for _ in range(3)]
    ref = oracle.residual_vjp(s, w.W0, alpha, dt, *bars)
    second, ratios, gks = sizes(s)
    tapes = ratios + (gks if s.flux == I.GKS else 0)
    # limit -> what a reverse holds under it, from the least to all, and back on the same handle
    steps = [(0, 0), (tapes - 1, 0), (tapes, tapes), (second + 2 * tapes - 1, tapes),
             (second + 2 * tapes, second + 2 * tapes), (None, second + 2 * tapes), (tapes, tapes), (0, 0)]
    with Solver(s) as sol:
        sol.set_reverse_memory(0)
        base = None
        for limit, held in steps:
            sol.set_reverse_memory(limit)
            got = adjoint_residual(sol, w.W0, alpha, dt, *bars)
            torch.cuda.synchronize()
            assert comp_rel_err(got.cpu().numpy(), ref) <= 1e-9, (limit, comp_rel_err(got.cpu().numpy(), ref))
            base = sol.device_bytes() if base is None else base
            assert sol.device_bytes() - base == held, (limit, sol.device_bytes() - base, held)


@pytest.mark.parametrize("flux", [I.GKS, I.LF])
def test_gradient_by_one_direction_at_a_time(flux):
    # records kept (read by a reverse of one direction at a time); then no second direction, no tapes
    from paper_2402_10914_gb300.solver import Solver, adjoint_steps
    w = I.random_smooth(18, 15, seed=57, flux=flux, time_limiter=1)
    s = w.settings
    dts = [0.4 * oracle.cfl_dt(s, w.W0) * f for f in (1.0, 0.9, 1.1)]
    WTb = np.random.default_rng(7).normal(size=w.W0.shape)
    _, ref = oracle.run_vjp(s, w.W0, dts, WTb)
    second = sizes(s)[0]
    with Solver(s) as sol:
        sol.set_reverse_memory(0)
        got = adjoint_steps(sol, w.W0, dts, WTb, ckpt_every=2)
        torch.cuda.synchronize()
        assert comp_rel_err(got.cpu().numpy(), ref) <= 1e-9
        held = sol.device_bytes()
        sol.set_reverse_memory(second)
        got = adjoint_steps(sol, w.W0, dts, WTb, ckpt_every=2)
        torch.cuda.synchronize()
        assert comp_rel_err(got.cpu().numpy(), ref) <= 1e-9
        assert sol.device_bytes() == held + second


@pytest.mark.parametrize("both", [False, True])
def test_ratio_tapes_without_the_flux_tapes(both):
    # room for an L-F reverse's tapes only: a GKS reverse then reads the ratios and evaluates its flux again
    from paper_2402_10914_gb300.solver import Solver, adjoint_residual
    w = I.random_rough(22, 19, seed=58, flux=I.LF, time_limiter=1)
    s = w.settings
    rng = np.random.default_rng(10)
    alpha = rng.uniform(0.0, 1.0, (s.ny, s.nx))
    dt = 0.4 * oracle.cfl_dt(s, w.W0)
    bars = [rng.normal(size=w.W0.shape) for _ in range(3)]
    second, ratios, _ = sizes(s)
    with Solver(s) as sol:
        sol.set_reverse_memory(second + 2 * ratios if both else ratios)
        for flux in (I.LF, I.GKS, I.LF):
            got = adjoint_residual(sol, w.W0, alpha, dt, *bars, flux=flux)
            torch.cuda.synchronize()
            held = sol.device_bytes() if flux == I.LF else held
            assert sol.device_bytes() == held
            ref = oracle.residual_vjp(s.with_(flux=flux), w.W0, alpha, dt, *bars)
            assert comp_rel_err(got.cpu().numpy(), ref) <= 1e-9
