"""What the reverse sweep holds on the device: tapes only where a reverse reads them, and only its flux's."""
import numpy as np
import pytest

import oracle
from paper_2402_10914_gb300 import inputs as I
from tests.parity_util import comp_rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NX, NY = 40, 32


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def tape_bytes(gks):
    # 6 values for each of a line's 8 and a face side's 4 reconstructions, 39 per Gauss point for the GKS flux,
    # in the larger direction's strides, for both directions
    up4 = lambda n: (n + 3) // 4 * 4  # noqa: E731
    lines = up4(max((NX + 1) * (NY + 4), (NY + 1) * (NX + 4)))
    sides = up4(2 * max((NX + 1) * NY, (NY + 1) * NX))
    return 2 * 8 * (48 * lines + 24 * sides + (39 * sides if gks else 0))


def case(flux):
    w = I.random_smooth(NX, NY, seed=31, flux=flux, time_limiter=1)
    rng = np.random.default_rng(3)
    return w, rng.uniform(0.2, 1.0, (NY, NX)), [rng.normal(size=w.W0.shape) for _ in range(3)]


def vjp(sol, w, alpha, bars):
    from paper_2402_10914_gb300.solver import adjoint_residual
    dt = 0.4 * oracle.cfl_dt(w.settings, w.W0)
    g = adjoint_residual(sol, w.W0, alpha, dt, *bars)
    torch.cuda.synchronize()
    return g.cpu().numpy(), oracle.residual_vjp(w.settings, w.W0, alpha, dt, *bars)


@pytest.mark.parametrize("flux", [I.GKS, I.LF])
def test_a_checkpointed_gradient_holds_no_tapes_of_its_own(flux):
    from paper_2402_10914_gb300.solver import Solver, adjoint_checkpointed, forward_checkpointed
    w, alpha, bars = case(flux)
    with Solver(w.settings) as sol:
        forward_checkpointed(sol, w.W0, 4, ckpt_every=2)
        adjoint_checkpointed(sol, bars[0])                  # reads the records that the forward pass kept
        held = sol.device_bytes()
        got, ref = vjp(sol, w, alpha, bars)                 # no records: evaluates its forward, with tapes
        assert sol.device_bytes() == held + tape_bytes(flux == I.GKS)
        assert comp_rel_err(got, ref) <= 1e-9
        held = sol.device_bytes()
        got, ref = vjp(sol, w, alpha, bars)                 # and keeps them
        assert sol.device_bytes() == held and comp_rel_err(got, ref) <= 1e-9


def test_the_flux_tapes_come_with_the_first_gks_reverse():
    from paper_2402_10914_gb300.solver import Solver, adjoint_residual
    w, alpha, bars = case(I.LF)
    dt = 0.4 * oracle.cfl_dt(w.settings, w.W0)
    with Solver(w.settings) as sol:
        got, ref = vjp(sol, w, alpha, bars)
        held = sol.device_bytes()
        assert comp_rel_err(got, ref) <= 1e-9
        g = adjoint_residual(sol, w.W0, alpha, dt, *bars, flux=I.GKS)
        torch.cuda.synchronize()
        ref = oracle.residual_vjp(w.settings.with_(flux=I.GKS), w.W0, alpha, dt, *bars)
        assert comp_rel_err(g.cpu().numpy(), ref) <= 1e-9
        assert sol.device_bytes() == held + tape_bytes(True) - tape_bytes(False)
        got, ref = vjp(sol, w, alpha, bars)                 # the other flux again, beside them
        assert comp_rel_err(got, ref) <= 1e-9


def test_a_captured_reverse_uses_what_is_there():
    # a reverse without records after a gradient, recorded into a graph: it must not allocate, so it runs untaped
    from paper_2402_10914_gb300.solver import Solver, adjoint_checkpointed, adjoint_residual, forward_checkpointed
    w, alpha, bars = case(I.GKS)
    dt = 0.4 * oracle.cfl_dt(w.settings, w.W0)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        Wd, ad, bd = dev(w.W0), dev(alpha), [dev(b) for b in bars]
        out = torch.zeros_like(Wd)
        with Solver(w.settings, stream=st) as sol:
            forward_checkpointed(sol, Wd, 4, ckpt_every=2)
            adjoint_checkpointed(sol, bd[0])
            held = sol.device_bytes()
            st.synchronize()
            graph = torch.cuda.CUDAGraph()
            graph.capture_begin(capture_error_mode="thread_local")
            adjoint_residual(sol, Wd, ad, dt, *bd, W_bar=out)
            graph.capture_end()
            assert sol.device_bytes() == held
            ref = oracle.residual_vjp(w.settings, w.W0, alpha, dt, *bars)
            for scale in (1.0, 0.5):
                for b, h in zip(bd, bars):
                    b.copy_(dev(scale * h))
                out.zero_()
                graph.replay()
                st.synchronize()
                assert comp_rel_err(out.cpu().numpy(), scale * ref) <= 1e-9
