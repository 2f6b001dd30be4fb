"""FP64 staged kernels at the edges of their thread map and of their fast paths.

One step against the oracle on batches of ragged cavities, below and above
the node count where the block size changes (32 and 128 threads), with
interiors that fill their last block by one lane, all of it, or a part; blends
eta_b = 1 and 0.3, lattice speed c = 2; and a zero-shear clamp so low that the
clamped argument of the power law lies beyond the exponents of its table.
Tolerances: those of the FP64 parity tests (1e-12, lambda's rounding bound).
"""
import numpy as np
import pytest

import oracle as O
from test_gpu_parity import cav, compare_state, lam_bound, solver
from test_gpu_parity_large import synthetic_state

pytestmark = pytest.mark.gpu

# interiors of 9, 476, 1024 = 32 x 32 and 129 = 4 x 32 + 1 nodes
SMALL = [(5, 5, 100.0, 0.75, 60.0), (9, 70, 100.0, 1.3, 45.0), (34, 34, 400.0, 0.6, 75.0),
         (45, 5, 100.0, 1.0, 90.0)]
LARGE = [(331, 307, 1000.0, 0.75, 60.0), (5, 9, 100.0, 1.25, 30.0), (66, 130, 400.0, 0.5, 60.0)]


def _check(specs, run_opts, opts, seed):
    runs = [O.cavity_run(sp[0], sp[2], sp[3], theta_deg=sp[4], ny=sp[1], **run_opts) for sp in specs]
    s = solver([cav(*sp) for sp in specs], kernel="staged", **opts)
    states = []
    for k, r in enumerate(runs):
        f0, l0 = (r.fhat.copy(), r.lam.copy()) if seed is None else synthetic_state(r, seed + 10 * k)
        s.set_state(k, f0, l0)
        states.append((f0, l0))
    s.step(1)
    res = s.residual()
    for k, (r, (f0, l0)) in enumerate(zip(runs, states)):
        fo, lo = O.step(f0, l0, r.g, r.prm)
        fg, lg = s.get_state(k)
        compare_state(fg, lg, fo, lo, lam_tol=lam_bound(f0, l0, r.prm, lo))
        Ek = O.kinetic_energy(*O.macros(fo)[:2], r.g)
        assert abs(res[k][3] - Ek) <= 1e-12 * Ek
    s.close()


@pytest.mark.parametrize("specs", [SMALL, LARGE], ids=["blocks of 32", "blocks of 128"])
@pytest.mark.parametrize("eta_b", [0.3, 1.0])
def test_ragged_batches(specs, eta_b):
    _check(specs, {"eta_b": eta_b}, {"eta_b": eta_b}, 300)


@pytest.mark.parametrize("gamma_min", [1e-60, 1e-20])
def test_clamp_beyond_the_power_table(gamma_min):
    """From rest f-hat equals f^eq exactly below the lid row, so that q = 0 is
    clamped at gamma_min^2 = 1e-120 (beyond a float's exponents: pow_fast) or
    1e-40: lambda is K gamma_min^(n-1) / c_s^2 to the power's error, 5e-16 +
    2.2e-16 |m log2 q| <= 1.2e-14 at m = -1/8, plus the reference's own."""
    r = O.cavity_run(37, 100.0, 0.75, theta_deg=60.0, ny=29, gamma_min=gamma_min)
    s = solver([cav(37, 29, 100.0, 0.75, 60.0)], kernel="staged", gamma_min=gamma_min)
    s.step(1)
    lam = s.get_state(0)[1][:-1]
    want = r.prm.K * gamma_min ** (0.75 - 1.0) * 3.0
    assert np.abs(lam - want).max() <= 2e-14 * want
    s.close()


def test_lattice_speed():
    """c = 2: the kernels' lattice units (u = c m, P = c_s^2 p) and speeds."""
    g = O.cavity_grid(37, 29, 1.0, 1.0, 60.0, 0.1, c=2.0)
    prm = O.cavity_params(37, 29, 100.0, 0.75, U=0.1, c=2.0, grid=g)
    f0, l0 = O.initial_state(g, prm)
    fo, lo = O.step(f0, l0, g, prm)
    s = solver([cav(37, 29, 100.0, 0.75, 60.0)], kernel="staged", c=2.0)
    s.step(1)
    fg, lg = s.get_state(0)
    compare_state(fg, lg, fo, lo, lam_tol=lam_bound(f0, l0, prm, lo))
    s.close()


def _adjoint_of(specs, states, weights):
    """One adjoint step of a batch: per cavity (adj_g, adj_lam) and dparams."""
    import torch

    from paper_2306_07603_gb300 import capi
    s = solver([cav(*sp) for sp in specs], kernel="staged", dt_mode="grid")

    def checkpoint(parts):
        for k, (f, lam) in enumerate(parts):
            s.set_state(k, f, lam)
        buf = torch.zeros(capi.ifdlbm_state_bytes(s.h) // 8 + 1, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        capi.ifdlbm_save_state_dev(s.h, buf)
        odd = buf[1:]                      # the same copy to an address off 16 bytes
        whole = buf.clone()
        torch.cuda.synchronize()
        capi.ifdlbm_save_state_dev(s.h, odd)
        s.sync()
        assert torch.equal(odd, whole[:-1])
        return whole[:-1].clone()

    adj, state = checkpoint(weights), checkpoint(states)
    dp = torch.zeros((len(specs), 3), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    capi.ifdlbm_adjoint_step(s.h, state, adj, dp)
    s.sync()
    out, planes = [], [sp[1] * ((sp[0] + 31) // 32 * 32) for sp in specs]
    g0, l0 = 0, 9 * sum(planes)
    for sp, p in zip(specs, planes):
        out.append((adj[g0:g0 + 9 * p].view(9, sp[1], -1)[:, :, :sp[0]].cpu().numpy(),
                    adj[l0:l0 + p].view(sp[1], -1)[:, :sp[0]].cpu().numpy()))
        g0, l0 = g0 + 9 * p, l0 + p
    s.close()
    return out, dp.cpu().numpy()


def test_adjoint_step_of_a_large_batch_equals_the_cavities_alone():
    """Blocks of 128 threads (above the node count of the one-warp blocks), a
    cluster per cavity in the reduction and ragged core and ring nodes: the
    adjoint of each small cavity equals its own in a handle of its own (blocks
    of one warp, which the dot-product and gradient tests hold to independent
    derivatives), to the rounding of the same operations: 1e-13 of the largest
    entry, and 1e-11 of the parameters' sums over some thousand terms."""
    specs = [(463, 441, 400.0, 0.75, 60.0), (5, 5, 100.0, 0.75, 60.0), (6, 40, 100.0, 1.25, 45.0),
             (37, 29, 400.0, 1.0, 90.0), (70, 7, 400.0, 0.6, 75.0)]
    runs = [O.cavity_run(sp[0], sp[2], sp[3], theta_deg=sp[4], ny=sp[1], dt_mode="grid")
            for sp in specs]
    states = [synthetic_state(r, 500 + 10 * k) for k, r in enumerate(runs)]
    weights = [synthetic_state(r, 900 + 10 * k) for k, r in enumerate(runs)]
    both, dp = _adjoint_of(specs, states, weights)
    for k in range(1, len(specs)):
        (one,), dp1 = _adjoint_of(specs[k:k + 1], states[k:k + 1], weights[k:k + 1])
        for a, b in zip(both[k], one):
            assert np.abs(a - b).max() <= 1e-13 * np.abs(b).max(), k
        assert np.all(np.abs(dp[k] - dp1[0]) <= 1e-11 * np.abs(dp1[0]) + 1e-300), k
