"""Free-stream preservation of the FP64 staged step: a uniform state stays uniform.

A cavity filled with fluid at rest and one pressure: the differences of a constant
are 0, so away from the walls (2 rows a stage, 4 a step) a step changes the
populations by the collision alone, which treats those of one speed alike. After
three steps the four populations of either speed are still equal there, at
every node and bit for bit; differences that leave their roundings behind separate
the populations that are advected along eta from those that are not.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("quad", [False, True])
def test_populations_of_one_speed_stay_equal(quad):
    import torch

    from paper_2306_07603_gb300 import capi
    from paper_2306_07603_gb300.solver import Solver, cavity, quad_cavity
    nx, ny, T = 65, 47, 3
    corners = ((0.0, 0.0), (1.0, 0.1), (-0.3, 1.0), (1.2, 0.9))
    cav = (quad_cavity(nx, ny, corners, 400.0, 0.75) if quad
           else cavity(nx, ny, 400.0, 0.75, theta_deg=60.0))
    Ps = np.random.default_rng(3).uniform(0.01, 0.5, 24)
    s = Solver([cav] * len(Ps))
    pitch, m = (nx + 31) // 32 * 32, 4 * T + 2
    wbar = np.array([-5 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
    # a state as saved: nine planes f-hat - w of every cavity, their relaxation times, their
    # reference pressures
    g = np.repeat(np.outer(Ps, wbar * 3.0).reshape(-1), ny * pitch)
    state = np.concatenate([g, np.full(len(Ps) * ny * pitch, 0.05), np.zeros(len(Ps))])
    buf = torch.tensor(state, device="cuda")
    assert buf.numel() * 8 == capi.ifdlbm_state_bytes(s.h)
    torch.cuda.synchronize()
    capi.ifdlbm_load_state_dev(s.h, buf)
    s.step(T)
    capi.ifdlbm_save_state_dev(s.h, buf)
    s.sync()
    g = buf.cpu().numpy()[:g.size].reshape(len(Ps), 9, ny, pitch)[:, :, m:-m, m:nx - m]
    s.close()
    for q in (2, 3, 4):
        assert np.array_equal(g[:, q], g[:, 1]), q
    for q in (6, 7, 8):
        assert np.array_equal(g[:, q], g[:, 5]), q
