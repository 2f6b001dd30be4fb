"""The fused step's automatic layout and overlapped launches.

Every node's arithmetic is the same in every layout, so the default one (rows
per task from the size of the batch, launches of consecutive steps overlapped
on small and on large grids) gives the state that other row counts and a
persistent schedule, whose launches do not overlap, give: to a rounding of the
largest population a step (different kernels may contract their operations
differently).
"""
import numpy as np
import pytest

from test_gpu_parity import cav, oracle_run, solver
from test_gpu_parity_large import synthetic_state

pytestmark = pytest.mark.gpu

# tasks of the default layout: few (overlapped), about one per SM, several per SM
# below and above four fifths of the slots (not overlapped, overlapped)
BATCHES = {
    "65x65": [(65, 65, 100.0, 0.75, 60.0)],
    "5x5 and 70x9": [(5, 5, 100.0, 0.75, 60.0), (70, 9, 100.0, 1.25, 45.0)],
    "129x129": [(129, 129, 400.0, 0.75, 60.0)],
    "10 of 129x257": [(129, 257, 400.0, 0.6, 75.0)] * 10,
    "11 of 257x257": [(257, 257, 1000.0, 1.4, 60.0)] * 11,
}
STEPS = 5


def _run(specs, states, **opts):
    s = solver([cav(*sp) for sp in specs], precision="fp32dev", kernel="fused", **opts)
    for k, (f, lam) in enumerate(states):
        s.set_state(k, f, lam)
    s.step(STEPS)
    out = [s.get_state(k) for k in range(len(specs))], s.residual()
    s.close()
    return out


@pytest.mark.parametrize("name", list(BATCHES))
def test_default_layout_equals_others(name):
    specs = BATCHES[name]
    one = synthetic_state(oracle_run(*specs[0]), 700)
    states = [one if sp == specs[0] else synthetic_state(oracle_run(*sp), 700 + k)
              for k, sp in enumerate(specs)]
    want, res = _run(specs, states)
    for opts in (dict(fused_rows=37, schedule="static"), dict(fused_threads=64, fused_rows=16)):
        got, r = _run(specs, states, **opts)
        for (fa, la), (fb, lb) in zip(got, want):
            assert np.abs(fa - fb).max() <= STEPS * 2.0 ** -23 * np.abs(fb - fb.mean()).max()
            assert np.abs(la - lb).max() <= 1e-3 * np.abs(lb).max()
        assert np.allclose(r, res, rtol=1e-5, atol=0.0)
