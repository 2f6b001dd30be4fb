"""The fused FP32 step's power of Eq. (1.4) is the rounded FP64 one, bit for bit.

The pairs of floats it is found in are within 2^-40 of the value; where the exact
value lies that close to the middle between two floats they may point to the wrong
one. Arguments: of 2^24 random ones those within 2^-36 of a middle (by a power good to
2^-52; about one in 2^12), where a plain rounding of the pair fails now and then,
2^18 of the others, and both ends of the exponents. n from 0.1 to 3, and beyond, where
FP64 has to take over. No tolerance: the two floats are equal.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [0.1, 0.5, 0.75, 1.25, 1.5, 3.0, 3.5, 8.0])
def test_every_float_is_the_rounded_fp64_one(n):
    import torch

    from paper_2306_07603_gb300 import capi
    from paper_2306_07603_gb300.solver import Solver, cavity
    s = Solver([cavity(9, 9, 400.0, n)], precision="fp32dev", kernel="fused")
    K = s.info(0).K
    rng = np.random.default_rng(11)
    x = (2.0 ** rng.uniform(-30, 20, 1 << 24)).astype(np.float32).astype(np.float64)
    want = K * 3 * x ** ((n - 1.0) / 2.0)
    f = want.astype(np.float32)
    gap = np.spacing(f).astype(np.float64)
    off = np.abs(want - f) / gap                                # 1/2: a middle between two floats
    near = np.abs(0.5 - off) * gap < 2.0 ** -36 * want
    assert near.sum() >= 1000 or n == 3.0   # (n = 3: C x = 3 x / 40 never comes close)
    x = np.concatenate([x[near], x[: 1 << 18], 2.0 ** np.arange(-126.0, 127.0)])
    xd = torch.tensor(x, device="cuda")
    out = torch.zeros(2 * len(x), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    capi.ifdlbm_selftest_pow_pair(s.h, 0, xd, out)
    s.sync()
    got, fp64 = out.cpu().numpy().reshape(2, -1)
    assert np.array_equal(got, fp64, equal_nan=True), np.sum(got != fp64)
    s.close()
