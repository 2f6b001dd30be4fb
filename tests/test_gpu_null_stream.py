"""Steps on the legacy default stream (stream NULL), whose launches overlap too.

The same cavities on a stream of their own give the same bits: in FP64 (three
overlapped kernels a step) and in the fused FP32 step, whose consecutive steps
overlap on a small grid; fields, a checkpoint and the residual follow on the stream.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,nx,ny", [("fp64", 65, 47), ("fp64", 130, 300), ("fp32dev", 65, 47)])
def test_default_stream_gives_the_same_bits(precision, nx, ny):
    import torch

    from paper_2306_07603_gb300 import capi
    from paper_2306_07603_gb300.solver import Solver, cavity, make_options

    def run(h, wait):
        nb = capi.ifdlbm_state_bytes(h)
        state = torch.zeros(nb // 8, dtype=torch.float64, device="cuda")
        psi = torch.zeros((ny, nx), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        capi.ifdlbm_step(h, 39)                      # a captured chunk and a remainder
        capi.ifdlbm_save_state_dev(h, state)
        capi.ifdlbm_macros_dev(h, 0, None, None, None, psi)
        wait()
        res = np.zeros((1, 4))
        capi.ifdlbm_batch_residual(h, res)
        return state.cpu(), psi.cpu(), torch.tensor(res)

    capi.use_torch_allocator()
    c = cavity(nx, ny, 400.0, 0.75, theta_deg=60.0)
    h = capi.ifdlbm_create_batch([c], make_options(precision=precision), 0)
    got = run(h, torch.cuda.synchronize)
    capi.ifdlbm_destroy(h)
    s = Solver([c], precision=precision)
    want = run(s.h, s.sync)
    s.close()
    for a, b in zip(got, want):
        assert torch.equal(a, b)
