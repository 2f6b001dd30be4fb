"""The FP64 staged kernels' power law (power64) against exact powers.

FP64 arguments over the table's exponents, on its cells' boundaries and beyond its
range on both sides, n up to 20. Bound (step64.cuh): four roundings, the rounding of
1/c_j times |m|, 1.5 half ulps of the FP32 tail coefficient b3 at |t| <= 2^-9, and the
first term of the series left out, |C(m,6)| 2^-54. Where the log2/exp2 form is to be
used instead (n > 3, or beyond the table) the value is that form's, bit for bit.
"""
import numpy as np
import pytest

from test_gpu_pow import _exact_power

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [0.05, 0.5, 0.75, 1.0, 1.5, 2.0, 3.0, 3.2, 5.0, 20.0])
def test_power64_relative_error(n):
    import torch

    from paper_2306_07603_gb300 import capi
    from paper_2306_07603_gb300.solver import Solver, cavity
    s = Solver([cavity(9, 9, 100.0, n)])
    C = s.info(0).K / (1.0 / 3.0)
    rng = np.random.default_rng(41)
    j = np.arange(256)
    edges = np.concatenate([1 + j / 256.0, 1 + (j + 0.5) / 256.0, np.nextafter(1 + (j + 1) / 256.0, 0)])
    x = np.concatenate([10.0 ** rng.uniform(-12, 8, 4000), edges, edges * 2.0 ** -20,
                        2.0 ** np.array([-126.0, -127.0, 127.0, 128.0, -200.0, 40.0])])
    xd = torch.tensor(x, device="cuda")
    out, fast, ref = (torch.zeros_like(xd) for _ in range(3))
    torch.cuda.synchronize()
    capi.ifdlbm_selftest_power64(s.h, 0, xd, out)
    capi.ifdlbm_selftest_pow(s.h, xd, (n - 1.0) / 2.0, fast, ref)
    s.sync()
    got = out.cpu().numpy()
    s.close()
    m = (n - 1.0) / 2.0
    want = _exact_power(x, m, C)
    b3, b6 = m * (m - 1) * (m - 2) / 6, m * (m - 1) * (m - 2) * (m - 3) * (m - 4) * (m - 5) / 720
    table = 4 * 2.0 ** -53 + 1.2e-16 * abs(m) + 1.5 * 2.0 ** -51 * abs(b3) + abs(b6) * 2.0 ** -54
    inside = (x >= 2.0 ** -126) & (x < 2.0 ** 128) & (abs(m) <= 1)
    assert np.array_equal(got[~inside], (C * fast.cpu().numpy())[~inside], equal_nan=True)
    rel = np.abs(got - want)[inside] / want[inside]
    bound = table + 2.0 ** -53                                    # (the reference's rounding)
    assert np.all(rel <= bound), (n, (rel / bound).max(), x[inside][np.argmax(rel)])
