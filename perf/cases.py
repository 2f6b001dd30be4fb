"""Timed cases of the IFDLBM library: the work its users have it do, through its public entry points.

A case is a dict of plain values:

  kind "step"      ``steps`` time steps of a batch of cavities (``Solver.step``), then the residuals
                   of the last step and a checkpoint of the whole state, read on the device
       "adjoint"   ``steps`` FP64 steps with their states and intermediates kept, then the reverse
                   sweep of the kinetic energy (the loop of the adjoint driver, nothing recomputed)
       "gradient"  the whole call ``energy_and_gradient``: n, Re, theta in, J and its gradient out
       "fields"    macroscopic fields, stream function, probes and the allocation-free residual
                   between two sets of fields, as a monitoring program reads them
  nx, ny, ncav     grid of the cavities and their number; with ``mix`` the cavities take 1, 3/4, 1/2
                   and 1/4 of the cells of that grid in turn
  precision        "fp64" or "fp32dev"; geometry "trapezoid" or "quad"; lambda_mode "lagged" or
                   "implicit"; threads, rows, schedule the fused step's layout (0, 0, "grid" = default)

The flow parameters (n, Re, theta or the corners) and the state are drawn from the seed: the state
is an equilibrium of smooth random P, u, v (|u| up to about half the lid speed) plus a smooth
non-equilibrium part, with a relaxation time around its value at unit shear rate, so that every node
carries gradients and shear. All handles of a process share one stream, as in a program that runs one
simulation after another (the allocation-free residual wants its calls serialised besides).
``exact`` is the scheme in plain FP64 torch, on the same inputs.
"""
import math

import numpy as np
import torch

from paper_2306_07603_gb300 import capi
from paper_2306_07603_gb300.adjoint import energy_and_gradient
from paper_2306_07603_gb300.solver import Solver, cavity, quad_cavity

_STEP = {"kind": "step", "precision": "fp32dev", "geometry": "trapezoid", "lambda_mode": "lagged",
         "mix": False, "threads": 0, "rows": 0, "schedule": "grid"}


def _step_case(name, nx, ny, ncav, steps, **more):
    return {**_STEP, "nx": nx, "ny": ny, "ncav": ncav, "steps": steps, **more, "name": name}


def listed():
    return [
        # the validation cavity, one small FP64 run: latency, launches, a chip mostly idle
        _step_case("fp64_cavity65", 65, 65, 1, 20, precision="fp64"),
        # the power-law sweep at the production grid in FP64 (reference runs, adjoint forward passes)
        _step_case("fp64_sweep257", 257, 257, 10, 4, precision="fp64"),
        # FP64 on general quadrilaterals, oblong odd-sized grids
        _step_case("fp64_quads193x129", 193, 129, 4, 6, precision="fp64", geometry="quad"),
        # the same validation cavity in FP32 deviations: one CUDA graph chunk and a remainder
        _step_case("fp32_cavity65", 65, 65, 1, 66),
        # the power-law sweep, the ordinary FP32 batch (its state stays in L2)
        _step_case("fp32_sweep257", 257, 257, 10, 33),
        # 64 uneven cavities in one launch, the benchmark's batch and layout (larger than L2)
        _step_case("fp32_batch64", 513, 513, 64, 12, mix=True, threads=128, rows=128,
                   schedule="dynamic"),
        # one large cavity, default layout (larger than L2)
        _step_case("fp32_single2049", 2049, 2049, 1, 9),
        # general quadrilaterals in FP32
        _step_case("fp32_quads257", 257, 257, 10, 20, geometry="quad"),
        # the implicit relaxation time, ragged grids
        _step_case("fp32_implicit300x260", 300, 260, 6, 10, lambda_mode="implicit"),
        # the reverse sweep of the adjoint at its production grid, everything kept
        {"kind": "adjoint", "nx": 257, "ny": 257, "steps": 6, "name": "adjoint257"},
        # a whole gradient with checkpoints, creation included
        {"kind": "gradient", "nx": 129, "ny": 129, "steps": 60, "every": 20, "name": "gradient129"},
        # fields, probes and residuals of three unsteady cavities
        {"kind": "fields", "nx": 1025, "ny": 1025, "ncav": 3, "precision": "fp32dev",
         "geometry": "trapezoid", "probes": 15, "name": "fields1025"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["adjoint", "gradient", "fields"])
    if kind == "adjoint":
        return {"kind": kind, "nx": _log_int(rng, 24, 400), "ny": _log_int(rng, 24, 400),
                "steps": rng.randint(2, 8)}
    if kind == "gradient":
        return {"kind": kind, "nx": _log_int(rng, 33, 140), "ny": _log_int(rng, 33, 140),
                "steps": rng.randint(20, 60), "every": rng.choice([1, 7, 20])}
    if kind == "fields":
        return {"kind": kind, "nx": _log_int(rng, 65, 1300), "ny": _log_int(rng, 65, 1300),
                "ncav": rng.randint(1, 3), "precision": rng.choice(["fp64", "fp32dev"]),
                "geometry": rng.choice(["trapezoid", "trapezoid", "quad"]),
                "probes": rng.randint(1, 40)}
    precision = rng.choice(["fp64", "fp32dev", "fp32dev"])
    mix = rng.random() < 0.3
    nodes = _log_int(rng, 3000, 400_000 if precision == "fp64" else 4_000_000)
    ncav = min(64, _log_int(rng, 1, 64))
    aspect = math.exp(rng.uniform(-0.7, 0.7))
    side = math.sqrt(max(nodes / ncav, 900.0))
    nx, ny = max(33 if mix else 5, int(side * aspect)), max(33 if mix else 5, int(side / aspect))
    return {**_STEP, "nx": nx, "ny": ny, "ncav": ncav, "mix": mix, "precision": precision,
            "geometry": rng.choice(["trapezoid", "trapezoid", "quad"]),
            "lambda_mode": rng.choice(["lagged", "lagged", "lagged", "implicit"]),
            "steps": rng.randint(1, 6) if precision == "fp64" else rng.randint(1, 40),
            "threads": rng.choice([0, 0, 64, 128, 256]), "rows": rng.choice([0, 0, 16, 37, 128]),
            "schedule": rng.choice(["grid", "grid", "static", "dynamic"])}


# ---------------------------------------------------------------- inputs from the seed

def _flows(case, seed):
    """Flow parameters of every cavity: nx, ny, n, Re, theta (or corners)."""
    rng = np.random.default_rng(seed)
    out = []
    for k in range(case.get("ncav", 1)):
        f = (1.0, 0.75, 0.5, 0.25)[k % 4] if case.get("mix") else 1.0
        nx, ny = (int((case[a] - 1) * f) + 1 for a in ("nx", "ny"))
        n = float(rng.uniform(0.5, 1.5))
        if case.get("lambda_mode") == "implicit":
            n = float(rng.choice([0.6, 0.75, 1.25, 1.4]))
        Re = float(rng.choice([100.0, 400.0, 1000.0] if min(nx, ny) >= 120 else [100.0, 200.0]))
        theta = float(rng.choice([45.0, 60.0, 75.0, 90.0]))
        d = rng.uniform(-0.2, 0.2, size=(4, 2))
        corners = None
        if case.get("geometry") == "quad":
            corners = tuple((float(x + d[i, 0]), float(y + d[i, 1]))
                            for i, (x, y) in enumerate(((0, 0), (1, 0), (0, 1), (1, 1))))
        out.append({"nx": nx, "ny": ny, "n": n, "Re": Re, "theta": theta, "corners": corners,
                    "implicit": case.get("lambda_mode") == "implicit", "grid_dt": False})
    return out


EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
WBAR = (-5 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
CS2 = 1.0 / 3.0
U_LID = 0.1


def _vec(v, like):
    return torch.tensor(v, dtype=torch.float64, device=like.device)[:, None, None]


def _noise(rng, ny, nx, amplitude):
    """A smooth random field: four Fourier modes."""
    x = torch.linspace(0.0, 1.0, nx, dtype=torch.float64, device="cuda")
    y = torch.linspace(0.0, 1.0, ny, dtype=torch.float64, device="cuda")
    out = torch.zeros((ny, nx), dtype=torch.float64, device="cuda")
    for _ in range(4):
        kx, ky = (int(v) for v in rng.integers(1, 4, size=2))
        px, py, a = (float(v) for v in (*rng.uniform(0, 2 * np.pi, size=2), rng.standard_normal()))
        out += a * torch.outer(torch.sin(np.pi * ky * y + py), torch.sin(np.pi * kx * x + px))
    return amplitude / 4 * out


def _state(flow, seed, k):
    """Deviations g = f-hat - w [9, ny, nx] and the lagged relaxation time [ny, nx], FP64."""
    rng = np.random.default_rng([seed, k])
    ny, nx = flow["ny"], flow["nx"]
    u, v, P = (_noise(rng, ny, nx, a) for a in (0.05, 0.05, 0.005))
    g = _feq(P, u, v)
    for q in range(9):
        g[q] += W[q] * _noise(rng, ny, nx, 4e-3)
    lam = _lam1(flow) * (1.0 + _noise(rng, ny, nx, 0.3))
    return g, lam


def _lam1(flow):
    """The relaxation time at unit shear rate."""
    return U_LID ** (2.0 - flow["n"]) / flow["Re"] / CS2


# ---------------------------------------------------------------- prepare and run

_stream = None


def _solver(flows, case):
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    if flows[0]["corners"]:
        cavs = [quad_cavity(f["nx"], f["ny"], f["corners"], f["Re"], f["n"], U_lid=U_LID)
                for f in flows]
    else:
        cavs = [cavity(f["nx"], f["ny"], f["Re"], f["n"], theta_deg=f["theta"], U_lid=U_LID)
                for f in flows]
    opts = {"precision": case["precision"], "stream": _stream}
    if flows[0]["implicit"]:
        opts["lambda_mode"] = "implicit"
    if flows[0]["grid_dt"]:
        opts.update(dt_mode="grid", kernel="staged")
    # the layout applies where the default choice of the kernel is the fused step
    if case["precision"] == "fp32dev" and case.get("threads"):
        opts["fused_threads"] = case["threads"]
    if case["precision"] == "fp32dev" and case.get("rows"):
        opts["fused_rows"] = case["rows"]
    if case["precision"] == "fp32dev" and case.get("schedule", "grid") != "grid":
        opts["schedule"] = case["schedule"]
    return Solver(cavs, **opts)


def _fill(s, flows, seed, precision):
    for k, f in enumerate(flows):
        g, lam = _state(f, seed, k)
        s.set_state(k, (g + _vec(W, g)).cpu().numpy(), lam.cpu().numpy())
    # a checkpoint holds the rows' padding too: start from one that has zeros there
    buf, at = _state_tensor(s, precision), 9 * _planes(flows)
    torch.cuda.synchronize()
    capi.ifdlbm_save_state_dev(s.h, buf)
    torch.cuda.synchronize()
    for f in flows:
        pitch = (f["nx"] + 31) // 32 * 32
        buf[at:at + f["ny"] * pitch].view(f["ny"], pitch)[:, f["nx"]:] = 0.0
        at += f["ny"] * pitch
    torch.cuda.synchronize()
    capi.ifdlbm_load_state_dev(s.h, buf)
    torch.cuda.synchronize()


def _state_tensor(s, precision):
    """A checkpoint buffer in the storage type: 10 planes per cavity, then one FP64 word each."""
    n = capi.ifdlbm_state_bytes(s.h)
    dtype = torch.float64 if precision == "fp64" else torch.float32
    return torch.zeros(n // dtype.itemsize, dtype=dtype, device="cuda")


def _planes(flows):
    return sum(f["ny"] * ((f["nx"] + 31) // 32 * 32) for f in flows)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "gradient":
        rng = np.random.default_rng(seed)
        return {"kind": kind, "args": (float(rng.uniform(0.7, 1.3)), float(rng.uniform(300, 500)),
                                       float(rng.uniform(50, 80)), case["nx"], case["ny"],
                                       case["steps"], case["every"])}
    if kind == "adjoint":
        case = {**case, "precision": "fp64"}
    flows = _flows(case, seed)
    if kind == "adjoint":
        flows[0]["grid_dt"] = True
    s = _solver(flows, case)
    _fill(s, flows, seed, case["precision"])
    st = {"kind": kind, "solver": s, "planes": _planes(flows)}
    if kind == "step":
        st["steps"], st["precision"] = case["steps"], case["precision"]
        st["state"] = _state_tensor(s, case["precision"])
        st["resid"] = torch.zeros((len(flows), 4), dtype=torch.float64, device="cuda")
    elif kind == "adjoint":
        st["steps"] = case["steps"]
        st["states"] = [_state_tensor(s, "fp64") for _ in range(case["steps"] + 1)]
        st["inter"] = [torch.empty(capi.ifdlbm_intermediate_bytes(s.h) // 8, dtype=torch.float64,
                                   device="cuda") for _ in range(case["steps"])]
        st["adj"] = _state_tensor(s, "fp64")
        st["dparams"] = torch.zeros(3, dtype=torch.float64, device="cuda")
        st["resid"] = torch.zeros((1, 4), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        capi.ifdlbm_save_state_dev(s.h, st["states"][0])
    else:
        shape = (flows[0]["ny"], flows[0]["nx"])
        st["fields"] = [[torch.zeros(shape, dtype=torch.float64, device="cuda") for _ in range(4)]
                        for _ in flows]
        st["pidx"], st["old"] = _field_inputs(case, flows, seed)
        st["pout"] = torch.zeros((case["probes"], 3), dtype=torch.float64, device="cuda")
        st["res"] = [torch.zeros(3, dtype=torch.float64, device="cuda") for _ in flows]
    torch.cuda.synchronize()
    return st


def _field_inputs(case, flows, seed):
    """Probe nodes, and the fields u, v, P of an earlier time."""
    rng = np.random.default_rng([seed, 77])
    ny, nx = flows[0]["ny"], flows[0]["nx"]
    idx = [(int(rng.integers(len(flows))), int(rng.integers(nx)), int(rng.integers(ny)))
           for _ in range(case["probes"])]
    old = [[_noise(rng, ny, nx, a) for a in (0.05, 0.05, 0.005)] for _ in flows]
    return torch.tensor(idx, dtype=torch.int32, device="cuda"), old


def run(state):
    kind = state["kind"]
    if kind == "gradient":
        n, Re, theta, nx, ny, T, every = state["args"]
        return list(energy_and_gradient(n, Re, theta, nx, ny, T, every=every))
    s, P = state["solver"], state["planes"]
    if kind == "step":
        s.step(state["steps"])
        capi.ifdlbm_residual_dev(s.h, state["resid"])
        capi.ifdlbm_save_state_dev(s.h, state["state"])
        resid = state["resid"]
        if state["precision"] != "fp64":     # the history of an FP32 run is kept in FP32
            with torch.cuda.stream(s.stream):
                resid = resid.float()
        return {"g": state["state"][:9 * P], "lam": state["state"][9 * P:10 * P], "resid": resid}
    if kind == "adjoint":
        states, inter, adj, dp = state["states"], state["inter"], state["adj"], state["dparams"]
        T = state["steps"]
        capi.ifdlbm_load_state_dev(s.h, states[0])
        for t in range(T):
            s.step(1)
            capi.ifdlbm_save_state_dev(s.h, states[t + 1])
            capi.ifdlbm_save_intermediates_dev(s.h, inter[t])
        capi.ifdlbm_residual_dev(s.h, state["resid"])
        with torch.cuda.stream(s.stream):
            dp.zero_()
        capi.ifdlbm_adjoint_seed_energy(s.h, states[T], adj, dp)
        for t in range(T - 1, -1, -1):
            capi.ifdlbm_adjoint_step_saved(s.h, states[t], states[t + 1], inter[t], adj, dp)
        return {"adj_g": adj[:9 * P], "adj_lam": adj[9 * P:10 * P], "dparams": dp,
                "energy": state["resid"][:, 3]}
    with torch.cuda.stream(s.stream):
        for k, (rho, u, v, psi) in enumerate(state["fields"]):
            capi.ifdlbm_macros_dev(s.h, k, rho, u, v, psi)
            p = (rho - 1.0) / 3.0
            u0, v0, p0 = state["old"][k]
            capi.ifdlbm_residual_fields_static(u.shape[1], u.shape[0], u, v, p, u0, v0, p0,
                                               state["res"][k], stream=s.stream.cuda_stream)
        capi.ifdlbm_probe_dev(s.h, state["pidx"], state["pout"])
    return {"fields": state["fields"], "residuals": state["res"], "probes": state["pout"]}


# ---------------------------------------------------------------- work

# flops of one node's step: two moment sets (25 each), two equilibria (70), power law and rates
# (30), three transforms (27 each), two mixed stencils (8 planes x 2 axes x 8) and the residual (20)
_FLOPS_STEP = 2 * 25 + 2 * 70 + 30 + 3 * 27 + 2 * 128 + 20


def work(case):
    if case["kind"] in ("adjoint", "gradient"):
        n = case["nx"] * case["ny"]
        # forward: state in and out. Reverse: state, f-bar^+ and f(t+dt/2), relaxation times
        # and the adjoint in, the adjoint out
        per = 160 + (10 + 18 + 1 + 10 + 10) * 8
        return {"bytes": n * case["steps"] * per, "flops": n * case["steps"] * 3 * _FLOPS_STEP}
    flows = _flows(case, 0)
    nodes = sum(f["nx"] * f["ny"] for f in flows)
    size = 8 if case["precision"] == "fp64" else 4
    if case["kind"] == "fields":             # nine planes in, four fields out, six fields in
        return {"bytes": nodes * (9 * size + 4 * 8 + 6 * 8), "flops": nodes * 45}
    # one step: ten planes in, ten out
    return {"bytes": nodes * case["steps"] * 20 * size, "flops": nodes * case["steps"] * _FLOPS_STEP}


# ---------------------------------------------------------------- the scheme in plain FP64 torch

def _moments(g):
    ex, ey = _vec(EX, g), _vec(EY, g)
    u, v = (ex * g).sum(0), (ey * g).sum(0)
    P = (CS2 / WBAR[0]) * (-g[1:].sum(0) + W[0] * (u * u + v * v) / (2 * CS2))
    return u, v, P


def _feq(P, u, v):
    w, wb, ex, ey = (_vec(t, u) for t in (W, WBAR, EX, EY))
    cu = ex * u + ey * v
    return wb * P / CS2 + w * (cu / CS2 + cu * cu / (2 * CS2 * CS2) - (u * u + v * v) / (2 * CS2))


def _metrics(flow, theta):
    """c_xi, c_eta [9, ny, nx], the Jacobian, x_eta, y_eta, dxi, deta."""
    nx, ny = flow["nx"], flow["ny"]
    xi = (torch.arange(nx, dtype=torch.float64, device="cuda") / (nx - 1))[None, :]
    eta = (torch.arange(ny, dtype=torch.float64, device="cuda") / (ny - 1))[:, None]
    one = torch.ones((ny, nx), dtype=torch.float64, device="cuda")
    if flow["corners"]:
        (x0, y0), (x1, y1), (x2, y2), (x3, y3) = flow["corners"]
    else:
        r = theta * (math.pi / 180.0)
        cot = torch.cos(r) / torch.sin(r)
        # bottom from cot to 1 + cot, lid from 0 to 1 + 2 cot
        x0, x1, x2, x3 = cot, 1.0 + cot, 0.0, 1.0 + 2.0 * cot
        y0, y1, y2, y3 = 0.0, 0.0, 1.0, 1.0
    x_xi = one * ((1 - eta) * (x1 - x0) + eta * (x3 - x2))
    y_xi = one * ((1 - eta) * (y1 - y0) + eta * (y3 - y2))
    x_eta = one * ((1 - xi) * (x2 - x0) + xi * (x3 - x1))
    y_eta = one * ((1 - xi) * (y2 - y0) + xi * (y3 - y1))
    J = x_xi * y_eta - x_eta * y_xi
    ex, ey = _vec(EX, J), _vec(EY, J)
    cxi = ex * (y_eta / J) + ey * (-x_eta / J)
    ceta = ex * (-y_xi / J) + ey * (x_xi / J)
    return cxi, ceta, J, x_eta, y_eta


def _mixed(F, c, dim, side):
    """The mixed difference (times 2 d) of all planes at the nodes where it is defined along `dim`."""
    n = F.shape[dim]

    def at(k, lo, hi):
        return F.narrow(dim, k + lo, n - 2 - lo - hi)

    f0, fm, fp = at(1, 0, 0), at(0, 0, 0), at(2, 0, 0)
    # far neighbours, extrapolated linearly beyond the walls
    fm2 = torch.cat([2 * F.narrow(dim, 0, 1) - F.narrow(dim, 1, 1), F.narrow(dim, 0, n - 3)], dim)
    fp2 = torch.cat([F.narrow(dim, 3, n - 3),
                     2 * F.narrow(dim, n - 1, 1) - F.narrow(dim, n - 2, 1)], dim)
    up = torch.where(side.narrow(dim, 1, n - 2), 3 * f0 - 4 * fm + fm2, -(3 * f0 - 4 * fp + fp2))
    return 0.5 * (fp - fm) + 0.5 * up


def _advect(F, m, nx, ny):
    """(c_xi D_xi + c_eta D_eta) F at the interior nodes [9, ny-2, nx-2]."""
    cxi, ceta = m[0], m[1]
    dx = _mixed(F, cxi, 2, cxi >= 0)[:, 1:-1, :] * (0.5 * (nx - 1))
    dy = _mixed(F, ceta, 1, ceta >= 0)[:, :, 1:-1] * (0.5 * (ny - 1))
    return cxi[:, 1:-1, 1:-1] * dx + ceta[:, 1:-1, 1:-1] * dy


def _walls(inner, flow):
    """All nodes [9, ny, nx] from the interior ones: walls by non-equilibrium extrapolation."""
    F = torch.nn.functional.pad(inner[None], (1, 1, 1, 1), mode="replicate")[0]
    u, v, P = _moments(F)
    uw, vw = torch.zeros_like(u), torch.zeros_like(v)
    if flow["corners"]:
        (_, _, (x2, y2), (x3, y3)) = flow["corners"]
        tl = math.hypot(x3 - x2, y3 - y2)
        lid = (U_LID * (x3 - x2) / tl, U_LID * (y3 - y2) / tl)
    else:
        lid = (U_LID, 0.0)
    uw[-1, 1:-1], vw[-1, 1:-1] = lid
    wall = torch.ones_like(u, dtype=torch.bool)
    wall[1:-1, 1:-1] = False
    return torch.where(wall, _feq(P, uw, vw) + (F - _feq(P, u, v)), F)


def _implicit_lambda(a, C, m, gmin, dt):
    """The root of lam = C max(a / (2 lam + dt), gmin)^m, by bisection and then Newton."""
    lamc = C * gmin ** m
    top = C * torch.clamp(a / dt, min=gmin) ** m
    lo = torch.zeros_like(a) if m < 0 else torch.full_like(a, lamc)
    hi = torch.full_like(a, lamc) if m < 0 else torch.maximum(top, lo)
    for _ in range(40):
        mid = 0.5 * (lo + hi)
        F = mid - C * torch.clamp(a / (2 * mid + dt), min=gmin) ** m
        lo, hi = torch.where(F > 0, lo, mid), torch.where(F > 0, mid, hi)
    lam = 0.5 * (lo + hi)
    for _ in range(4):
        Pw = C * torch.clamp(a / (2 * lam + dt), min=gmin) ** m
        lam = lam - (lam - Pw) / (1 + 2 * m * Pw / (2 * lam + dt))
    return torch.where(a <= gmin * (2 * lamc + dt), torch.full_like(a, lamc), lam)


def _one_step(g, lam_prev, flow, n, Re, m, dt):
    gmin = 1e-3 * U_LID
    C = U_LID ** (2.0 - n) / Re / CS2
    u, v, P = _moments(g)
    feq = _feq(P, u, v)
    ex, ey = _vec(EX, g), _vec(EY, g)
    d = g - feq
    pxx, pxy, pyy = (ex * ex * d).sum(0), (ex * ey * d).sum(0), (ey * ey * d).sum(0)
    pp = 0.5 * (pxx * pxx + 2 * pxy * pxy + pyy * pyy)
    if flow["implicit"]:
        lam = _implicit_lambda(2 * torch.sqrt(pp) / CS2, C, n - 1.0, gmin, dt)
    else:
        k = -2.0 / ((2 * lam_prev + dt) * CS2)
        lam = C * torch.clamp(k * k * pp, min=gmin * gmin) ** (0.5 * (n - 1.0))
    i2 = 1.0 / (2 * lam + dt)
    fp, fb = g + 2 * dt * i2 * (feq - g), g + 1.5 * dt * i2 * (feq - g)
    nx, ny = flow["nx"], flow["ny"]
    fbar = fb[:, 1:-1, 1:-1] - 0.5 * dt * _advect(fb, m, nx, ny)
    bu, bv, bP = _moments(fbar)
    bh = (dt / (4 * lam + dt))[1:-1, 1:-1]
    fh = _walls(fbar + bh * (_feq(bP, bu, bv) - fbar), flow)
    return _walls(fp[:, 1:-1, 1:-1] - dt * _advect(fh, m, nx, ny), flow), lam, (u, v, P)


def _time_step(flow):
    nx, ny = flow["nx"], flow["ny"]
    if flow["grid_dt"]:
        return 0.5 * min(1.0 / (nx - 1), 1.0 / (ny - 1))
    cxi, ceta = _metrics(flow, torch.tensor(flow["theta"], dtype=torch.float64, device="cuda"))[:2]
    return 0.5 * min(1.0 / (nx - 1) / float(cxi.abs().max()),
                     1.0 / (ny - 1) / float(ceta.abs().max()))


def _weights(flow):
    wx = torch.full((flow["nx"],), 1.0 / (flow["nx"] - 1), dtype=torch.float64, device="cuda")
    wy = torch.full((flow["ny"],), 1.0 / (flow["ny"] - 1), dtype=torch.float64, device="cuda")
    for w in (wx, wy):
        w[0] *= 0.5
        w[-1] *= 0.5
    return wy[:, None] * wx[None, :]


def _residual(new, old, J, w):
    (u1, v1, P1), (u0, v0, P0) = new, old
    du2 = (u1 - u0) ** 2 + (v1 - v0) ** 2
    u2 = u1 * u1 + v1 * v1
    return [float(torch.sqrt(du2.sum() / u2.sum())),
            float(torch.sqrt(((P1 - P0) ** 2).sum() / (P1 * P1).sum())),
            float(torch.sqrt(du2.max() / u2.max())), float((0.5 * u2 * J * w).sum())]


def _padded(F, flow):
    pitch = (flow["nx"] + 31) // 32 * 32
    return torch.nn.functional.pad(F, (0, pitch - flow["nx"])).reshape(-1)


def _exact_step(case, seed):
    gs, lams, res = [], [], []
    for k, flow in enumerate(_flows(case, seed)):
        g, lam = _state(flow, seed, k)
        m = _metrics(flow, torch.tensor(flow["theta"], dtype=torch.float64, device="cuda"))
        dt = _time_step(flow)
        for _ in range(case["steps"]):
            g, lam, old = _one_step(g, lam, flow, flow["n"], flow["Re"], m, dt)
        res.append(_residual(_moments(g), old, m[2], _weights(flow)))
        gs.append(_padded(g, flow))
        lams.append(_padded(lam, flow))
    return {"g": torch.cat(gs), "lam": torch.cat(lams),
            "resid": torch.tensor(res, dtype=torch.float64, device="cuda")}


def _energy(g, m, flow):
    u, v, _ = _moments(g)
    return (0.5 * (u * u + v * v) * m[2] * _weights(flow)).sum()


def _leaf(v):
    return torch.tensor(float(v), dtype=torch.float64, device="cuda", requires_grad=True)


def _exact_adjoint(case, seed):
    flow = {**_flows(case, seed)[0], "grid_dt": True}
    g0, lam0 = _state(flow, seed, 0)
    g, lam = g0.clone().requires_grad_(True), lam0.clone().requires_grad_(True)
    n, Re, theta = _leaf(flow["n"]), _leaf(flow["Re"]), _leaf(flow["theta"])
    m, dt = _metrics(flow, theta), _time_step(flow)
    a, b = g, lam
    for _ in range(case["steps"]):
        a, b, _ = _one_step(a, b, flow, n, Re, m, dt)
    J = _energy(a, m, flow)
    ag, al, *dp = torch.autograd.grad(J, (g, lam, n, Re, theta))
    return {"adj_g": _padded(ag, flow), "adj_lam": _padded(al, flow), "dparams": torch.stack(dp),
            "energy": J.detach().reshape(1)}


def _exact_gradient(case, seed):
    n0, Re0, theta0, nx, ny, T, _ = prepare(case, seed)["args"]
    flow = {"nx": nx, "ny": ny, "n": n0, "Re": Re0, "theta": theta0, "corners": None,
            "implicit": False, "grid_dt": True}
    n, Re, theta = _leaf(n0), _leaf(Re0), _leaf(theta0)
    m, dt = _metrics(flow, theta), _time_step(flow)
    rest = torch.zeros((ny, nx), dtype=torch.float64, device="cuda")
    uw = rest.clone()
    uw[-1, 1:-1] = U_LID
    g = _feq(rest, uw, rest)
    lam = U_LID ** (2.0 - n) / Re / CS2 * (1e-3 * U_LID) ** (n - 1.0) * torch.ones_like(rest)
    lam = lam.detach()      # f^ne is 0 at rest: the first relaxation time does not enter
    for _ in range(T):
        g, lam, _ = _one_step(g, lam, flow, n, Re, m, dt)
    J = _energy(g, m, flow)
    return [float(J), *(float(v) for v in torch.autograd.grad(J, (n, Re, theta)))]


def _exact_fields(case, seed):
    flows = _flows(case, seed)
    pidx, old = _field_inputs(case, flows, seed)
    fields, res, macros = [], [], []
    for k, flow in enumerate(flows):
        g, _ = _state(flow, seed, k)
        u, v, P = _moments(g)
        macros.append((u, v, P))
        m = _metrics(flow, torch.tensor(flow["theta"], dtype=torch.float64, device="cuda"))
        I = u * m[4] - v * m[3]
        psi = torch.zeros_like(I)
        psi[1:] = torch.cumsum(0.5 * (I[1:] + I[:-1]) / (flow["ny"] - 1), 0)
        fields.append([1.0 + 3.0 * P, u, v, psi])
        r = _residual((u, v, P), old[k], m[2], _weights(flow))
        res.append(torch.tensor(r[:3], dtype=torch.float64, device="cuda"))
    probes = torch.stack([torch.stack([f[j, i] for f in macros[c]]) for c, i, j in pidx.tolist()])
    return {"fields": fields, "residuals": res, "probes": probes}


def exact(case, seed):
    return {"step": _exact_step, "adjoint": _exact_adjoint, "gradient": _exact_gradient,
            "fields": _exact_fields}[case["kind"]](case, seed)
