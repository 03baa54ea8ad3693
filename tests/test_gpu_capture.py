"""Stage operators recorded into a CUDA graph: their kernels are launched ahead of their predecessor's end, so a
capture records programmatic edges, and a replay on new inputs must give what a direct call gives, bit for bit.
(dfgks_residual_noalloc one direction after the other, dfgks_residual both at once; meshes on either side of the
line to four threads per item.)"""
import ctypes as C

import numpy as np
import pytest

from paper_2402_10914_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = {
    "quadrants_96": lambda: I.quadrants(96, seed=3),
    "limit_128": lambda: I.random_smooth(128, 128, seed=8, flux=I.GKS),
    "rough_23x17_lf": lambda: I.random_rough(23, 17, seed=6, bc=(I.PERIODIC, I.PERIODIC, I.REFLECT, I.OUTFLOW),
                                             flux=I.LF, time_limiter=0),
    "one_cell": lambda: I.random_rough(1, 1, seed=5, flux=I.GKS),
}


def p(t):
    return C.c_void_p(t.data_ptr())


@pytest.mark.parametrize("entry", ["noalloc", "handle"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_replays_equal_direct_calls(name, entry):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2402_10914_gb300 import _lib
    from paper_2402_10914_gb300.solver import Solver, make_config
    w = CASES[name]()
    s = w.settings
    st = torch.cuda.Stream()
    rng = np.random.default_rng(2)
    with torch.cuda.stream(st), Solver(s, stream=st) as sol:
        W = torch.as_tensor(w.W0, dtype=torch.float64, device="cuda").contiguous()
        alpha = torch.as_tensor(rng.uniform(0.0, 1.0, (s.ny, s.nx)), device="cuda")
        out = [torch.empty_like(W) for _ in range(3)] + [torch.empty_like(alpha)]
        cfg = make_config(s)

        def call():
            args = (p(W), p(alpha), 1e-3, int(s.flux), *[p(o) for o in out])
            rc = _lib.lib().dfgks_residual_noalloc(C.byref(cfg), C.c_void_p(st.cuda_stream), *args) if entry == "noalloc" \
                else _lib.lib().dfgks_residual(sol._h, *args)
            assert rc == _lib.OK, _lib.status_string(rc)

        call()                                   # the first call looks the scratch array up, outside a capture
        st.synchronize()
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin(capture_error_mode="thread_local")
        call()
        graph.capture_end()
        for k in range(3):
            W.copy_(torch.as_tensor(w.W0 * (1.0 + 0.01 * k)))
            alpha.copy_(torch.as_tensor(rng.uniform(0.0, 1.0, (s.ny, s.nx))))
            call()
            st.synchronize()
            direct = [o.clone() for o in out]
            for o in out:
                o.fill_(float("nan"))
            for _ in range(2):
                graph.replay()
            st.synchronize()
            for a, b in zip(out, direct):
                assert torch.equal(a, b), (name, entry, k)
