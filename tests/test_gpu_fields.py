"""Fields and stream function against the oracle, on both sides of the height from which
a cluster of blocks shares the lines (256 rows), for trapezoids and quadrilaterals.

Bounds, g being the deviations f-hat - w of the state and eps the storage's: storing g
and adding six (u, v) or eight (P) of it leaves 16 eps max|g| on u and v and
40 eps max|g| on the sum of Eq. (2.11), 72 eps max|g| on rho = rho0 + 3 P; in FP64
the state comes as f-hat, whose rounding counts besides (max|f-hat| for max|g|). psi
integrates u y_eta - v x_eta over the unit height: their error, and one rounding of
the sum per row.
"""
import numpy as np
import pytest

import oracle as O
from test_gpu_parity import cav, solver
from test_gpu_parity_large import synthetic_state

pytestmark = pytest.mark.gpu
CORNERS = ((0.0, 0.0), (1.0, 0.1), (-0.3, 1.0), (1.2, 0.9))


@pytest.mark.parametrize("precision", ["fp64", "fp32dev"])
@pytest.mark.parametrize("quad", [False, True])
@pytest.mark.parametrize("nx,ny", [(47, 255), (64, 256), (33, 257), (70, 600), (300, 1025)])
def test_fields_and_stream_function(nx, ny, quad, precision):
    from paper_2306_07603_gb300.solver import Solver, quad_cavity
    if quad:
        run = O.quad_run(nx, ny, CORNERS, 400.0, 0.75)
        s = Solver([quad_cavity(nx, ny, CORNERS, 400.0, 0.75)], precision=precision)
    else:
        run = O.cavity_run(nx, 400.0, 0.75, theta_deg=60.0, ny=ny)
        s = solver([cav(nx, ny, 400.0, 0.75, 60.0)], precision=precision)
    f, lam = synthetic_state(run, 60)
    s.set_state(0, f, lam)
    got = s.macros(0)
    s.close()
    u, v, P = O.macros(f)
    g = np.abs(f if precision == "fp64" else f - O.OMEGA[:, None, None]).max()
    eps = np.finfo(np.float64 if precision == "fp64" else np.float32).eps
    eu, er = 16 * eps * g, 72 * eps * g
    assert np.abs(got["u"] - u).max() <= eu and np.abs(got["v"] - v).max() <= eu
    assert np.abs(got["rho"] - (1.0 + 3.0 * P)).max() <= er
    psi = O.stream_function(u, v, run.g)
    slope = max(np.abs(run.g.y_eta).max(), np.abs(run.g.x_eta).max())
    bound = 2 * slope * eu + ny * np.finfo(float).eps * 2 * slope * max(np.abs(u).max(), np.abs(v).max())
    assert np.abs(got["psi"] - psi).max() <= bound
    assert (got["psi"][0] == 0).all()
