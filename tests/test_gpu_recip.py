"""The FP64 kernels' reciprocal against the division.

Bound: one rounding, plus the cube of the FP32 seed's relative error (2^-23 for the
truncated argument and 2^-22 for two ulps of the FP32 quotient: 2^-64.2, 2^-11 of an
ulp), with 2^-11 ulp more for the extended-precision reference of the host. Against
the rounded division at most one argument in 2^9 differs (two in 2^11 of the
distance between two doubles lie that close to a middle), by one ulp. Outside
[2^-100, 2^100), and for zeros, negative numbers, infinities and NaN: the division.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_recip_is_the_division_to_half_an_ulp():
    import torch

    from paper_2306_07603_gb300 import capi
    from paper_2306_07603_gb300.solver import Solver, cavity
    s = Solver([cavity(9, 9, 100.0, 0.75)])
    rng = np.random.default_rng(5)
    cells = 1.0 + np.arange(4096) / 4096.0
    x = np.concatenate([2.0 ** rng.uniform(-100, 100, 200_000), 2.0 ** rng.uniform(-30, 30, 200_000),
                        cells, np.nextafter(cells, 0), np.nextafter(cells, 4), 2.0 ** np.arange(-100.0, 100.0)])
    beyond = np.array([0.0, -0.0, 1e-320, 2.0 ** -101, 2.0 ** 100, 1e300, np.inf, -np.inf, np.nan, -3.7,
                       -1e-200, 2.0 ** -1022, np.nextafter(2.0 ** -100, 0)])
    xd = torch.tensor(np.concatenate([x, beyond]), device="cuda")
    out = torch.zeros_like(xd)
    torch.cuda.synchronize()
    capi.ifdlbm_selftest_recip(s.h, xd, out)
    s.sync()
    got, other = np.split(out.cpu().numpy(), [x.size])
    s.close()
    with np.errstate(divide="ignore", over="ignore"):
        assert np.array_equal(other, 1.0 / beyond, equal_nan=True)
    want = 1.0 / np.longdouble(x)
    ulp = np.spacing(want.astype(np.float64))
    err = (np.abs(np.longdouble(got) - want) / ulp).astype(np.float64)
    assert err.max() <= 0.5 + 2.0 ** -10, (err.max(), x[err.argmax()])
    assert np.mean(got != 1.0 / x) <= 2.0 ** -9
