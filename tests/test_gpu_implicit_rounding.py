"""The implicit relaxation time of the fused FP32 step is the FP64 root, rounded.

The FP64 solve knows F = lambda - P to about 1.6e-15 of lambda and the root to
1/min(1, n) of that, so that its float differs from the exact root's for up to
0.053/min(1, n) roots in 10^6 (twice the error over the least spacing of floats, 6e-8
of the value): 2 + three times as many may differ, by one ulp. One Newton step in
pairs of floats from an approximate root, rounded without looking whether it settles
the float, misses some tens for small n and large relaxation times, where the
approximation's error is amplified most. n over the range, shear rates from the clamp on.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", [1e-4, 2e-3, 3e-2])
@pytest.mark.parametrize("n", [0.01, 0.05, 0.3, 0.75, 1.0, 1.4, 2.5, 3.0, 4.0])
def test_every_root_is_the_rounded_fp64_one(n, dt):
    import torch

    from paper_2306_07603_gb300 import capi
    from paper_2306_07603_gb300.solver import Solver, cavity
    s = Solver([cavity(9, 9, 400.0, n)], precision="fp32dev", kernel="fused",
               lambda_mode="implicit", dt=dt)
    info = s.info(0)
    rng = np.random.default_rng(23)
    gam = info.gamma_min * 10.0 ** rng.uniform(-0.3, 5.5, 1_000_000)
    lam = 3.0 * info.K * gam ** (n - 1.0)
    G2 = (gam * (2.0 * lam + dt) / 6.0) ** 2
    x = torch.tensor(np.concatenate([G2, lam * rng.uniform(0.5, 1.5, gam.size)]), device="cuda")
    out = torch.zeros(2 * gam.size, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    capi.ifdlbm_selftest_implicit(s.h, 0, x, out)
    s.sync()
    got, fp64 = out.cpu().numpy().reshape(2, -1)
    assert np.isfinite(fp64).all()
    differ = got != fp64
    assert differ.sum() <= 2 + 0.16 / min(1.0, n), differ.sum()
    assert (np.abs(got - fp64)[differ] <= 1.5 * np.spacing(fp64[differ].astype(np.float32))).all()
    s.close()
