"""The FP32 step's power of Eq. (1.4) in pairs of floats (ifdlbm_selftest_pow_pair).

Every term is carried to 2^-40 of the result before one rounding to FP32, so
that the value may miss the nearest float only where the exact one lies within
2^-40 (2^-16 ulp) of a rounding boundary: the error stays within 0.5 ulp + 1e-4
ulp (the bound taken here, with the table entries' own 2^-48 and a factor 6 of
room), and against the rounded FP64 evaluation at most one argument in 2^13 may
differ, by one ulp (one in 2^16 expected). Reference: NumPy's extended
precision. n from 0.1 to 3; arguments over the exponents the clamp leaves, on
the table's cell boundaries, and, for n = 3, on both sides of the range the
table covers (beyond it the FP64 evaluation takes over).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [0.1, 0.5, 0.75, 1.0, 1.25, 1.5, 3.0])
def test_pow_pair_is_the_nearest_float(n):
    import torch

    from paper_2306_07603_gb300 import capi
    from paper_2306_07603_gb300.solver import Solver, cavity
    s = Solver([cavity(9, 9, 400.0, n)], precision="fp32dev", kernel="fused")
    info = s.info(0)
    rng = np.random.default_rng(7)
    cells = (1.0 + np.arange(256) / 256.0)
    x = np.concatenate([2.0 ** rng.uniform(-40, 40, 200_000), cells, np.nextafter(
        cells.astype(np.float32), np.float32(0)), 2.0 ** np.arange(-126.0, 127.0)])
    xf = x.astype(np.float32).astype(np.float64)
    xd = torch.tensor(xf, device="cuda")
    out = torch.zeros(2 * len(xf), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    capi.ifdlbm_selftest_pow_pair(s.h, 0, xd, out)
    s.sync()
    got, tab = out.cpu().numpy().reshape(2, -1)
    C = np.longdouble(info.K) / (np.longdouble(1.0) / 3)
    want = C * np.longdouble(xf) ** np.longdouble((n - 1.0) / 2.0)
    normal = (want > 2.0 ** -120) & (want < 2.0 ** 120)
    ulp = np.spacing(np.abs(want[normal]).astype(np.float32)).astype(np.float64)
    err = np.abs(got[normal] - want[normal]).astype(np.float64) / ulp
    assert err.max() <= 0.5 + 1e-4, err.max()
    differ = got != tab
    assert differ.mean() <= 2.0 ** -13, differ.mean()
    assert np.all(np.abs(got - tab)[differ & normal] <= 1.5 * ulp[differ[normal]])
    s.close()
