"""The implicit relaxation time's solves over their ranges.

One step of the FP32 form (FP32 root, one Newton step in pairs of floats) and of
the FP64 form (the same root as the start of the FP64 iteration) against the
oracle's bisection, for n from 0.3 to 2.5, with the clamp below every node's
shear rate, above about half of them, and far outside a float's range (where
the FP64 form starts from the lagged value).

Bound on lambda: it is C gamma(lambda)^(n-1), gamma = a / (2 lambda + dt), so a
relative error of a is amplified by at most |n - 1| / min(1, n); a comes from
second moments of f-hat - f^eq, whose rounding is taken as 16 eps max|g| (as in
the other parity tests), plus 1e-6 (FP32) or 1e-12 (FP64) of the largest lambda.
"""
import numpy as np
import pytest

import oracle as O
from test_gpu_parity import cav, solver
from test_gpu_parity_large import synthetic_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32dev", "fp64"])
@pytest.mark.parametrize("gamma_min", [1e-4, 0.3, 1e-60])
@pytest.mark.parametrize("n", [0.3, 0.6, 1.4, 2.5])
def test_implicit_lambda_over_its_range(n, gamma_min, precision):
    if gamma_min < 1e-30 and precision == "fp32dev":
        pytest.skip("the FP32 form clamps its FP32 strain rate at a normal float")
    nx, ny = 61, 47
    run = O.cavity_run(nx, 100.0, n, theta_deg=60.0, ny=ny, implicit_lambda=True,
                       gamma_min=gamma_min)
    f0, l0 = synthetic_state(run, 40)
    l0 = np.clip(l0, 1e-6, 10.0)
    fo, lo = O.step(f0, l0, run.g, run.prm)
    s = solver([cav(nx, ny, 100.0, n, 60.0)], precision=precision, lambda_mode="implicit",
               gamma_min=gamma_min)
    s.set_state(0, f0, l0)
    s.step(1)
    lg = s.get_state(0)[1]
    s.close()
    ux, uy, P = O.macros(f0)
    d = f0 - O.equilibrium(P, ux, uy)
    ex, ey = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1]), np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])
    pxx, pxy, pyy = (np.tensordot(c, d, 1) for c in (ex * ex, ex * ey, ey * ey))
    size = np.sqrt(0.5 * (pxx ** 2 + 2 * pxy ** 2 + pyy ** 2))
    g = f0 - O.OMEGA[:, None, None]
    eps, floor = (np.finfo(np.float32).eps, 1e-6) if precision == "fp32dev" else \
        (np.finfo(float).eps, 1e-12)
    noise = 16 * eps * np.abs(g if precision == "fp32dev" else f0).max() / size
    bound = abs(n - 1) / min(1.0, n) * lo * noise + floor * np.abs(lo).max()
    assert np.all(np.abs(lg - lo) <= bound), np.max(np.abs(lg - lo) / bound)
