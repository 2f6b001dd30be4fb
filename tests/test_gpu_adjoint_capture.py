"""A first adjoint call inside a graph capture leaves the handle usable.

A captured call executes nothing, so the tables it would form (which block belongs to
which cavity among them) are not there for a call outside the graph, which has
to form them itself; and the graph forms them for its own replays.
"""
import pytest

pytestmark = pytest.mark.gpu


def test_first_adjoint_call_captured_then_called_directly():
    import torch

    from paper_2306_07603_gb300 import capi
    from paper_2306_07603_gb300.solver import Solver, cavity

    def handle():
        s = Solver([cavity(67, 45, 400.0, 0.75, theta_deg=60.0)], kernel="staged", dt_mode="grid")
        s.step(20)
        new = lambda n: torch.zeros(n // 8, dtype=torch.float64, device="cuda")  # noqa: E731
        b = {"s0": new(capi.ifdlbm_state_bytes(s.h)), "s1": new(capi.ifdlbm_state_bytes(s.h)),
             "in": new(capi.ifdlbm_intermediate_bytes(s.h)), "adj": new(capi.ifdlbm_state_bytes(s.h)),
             "dp": new(24)}
        torch.cuda.synchronize()
        capi.ifdlbm_save_state_dev(s.h, b["s0"])
        s.step(1)
        capi.ifdlbm_save_state_dev(s.h, b["s1"])
        capi.ifdlbm_save_intermediates_dev(s.h, b["in"])
        s.sync()
        return s, b

    def sweep(s, b):
        with torch.cuda.stream(s.stream):
            b["adj"].zero_()
            b["dp"].zero_()
        capi.ifdlbm_adjoint_seed_energy(s.h, b["s1"], b["adj"], b["dp"])
        capi.ifdlbm_adjoint_step_saved(s.h, b["s0"], b["s1"], b["in"], b["adj"], b["dp"])

    def result(s, b):
        s.sync()
        return b["adj"].clone(), b["dp"].clone()

    ref, rb = handle()
    sweep(ref, rb)
    want = result(ref, rb)
    s, b = handle()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s.stream):
        sweep(s, b)                        # recorded, not run
    for run in (lambda: sweep(s, b), graph.replay, lambda: sweep(s, b)):
        with torch.cuda.stream(s.stream):
            run()
        got = result(s, b)
        assert all(torch.equal(x, y) for x, y in zip(got, want))
    ref.close()
    s.close()
