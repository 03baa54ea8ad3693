"""A decomposition's block table goes to the device in the order of the stream that reads it.

A copy from pageable memory on the legacy stream may return before the data has arrived, and streams that
are not blocking (the handle's own, a caller's torch.cuda.Stream) do not wait for the legacy stream."""
import os
import re

import numpy as np
import pytest

from paper_2402_10914_gb300 import inputs as I

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_10914_gb300", "csrc")


def test_every_upload_names_its_stream():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh", ".h")):
            text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
            for call in re.findall(r"\bcudaMemcpy(?:2D|ToSymbol)?\s*\([^;]*;", text):
                assert "HostToDevice" not in call, (f, call)


@pytest.mark.gpu
def test_steps_right_after_creation_on_a_caller_stream():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    from paper_2402_10914_gb300.solver import DecompSolver, Solver
    __graft_entry__.build()
    w = I.quadrants(48, seed=3)
    with Solver(w.settings) as s:
        s.set_ic(w.W0)
        s.step(2)
        W, a, t, _ = s.get_state()
    busy = torch.zeros(1 << 26, dtype=torch.float64, device="cuda")
    for _ in range(3):
        for _ in range(20):
            busy.add_(1.0)                     # the legacy stream has work of its own meanwhile
        with DecompSolver(w.settings, 3, 2, stream=torch.cuda.Stream()) as d:
            d.set_ic(w.W0)
            assert d.step(2) == 2
            Wd, ad, td, _ = d.get_state()
        assert np.array_equal(W, Wd) and np.array_equal(a, ad) and t == td
