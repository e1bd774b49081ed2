"""Performance cases: what a user of this framework has it do, one public call path per case.

A case is a dict of plain values.  listed() holds the fixed cases, draw(rng) makes one more of
the same ranges, prepare(case, seed) builds what a program has in hand before the call (inputs
on the GPU and the handle it keeps), run(state) is one pass and returns its outputs,
work(case) the bytes and operations a pass cannot do without, and exact(case, seed) the same
outputs in 64 bits from plain torch.

Kinds of case:
  grid      one SEIRD grid: write the state, advance it, read it back (and, with "diag", the
            population totals and the peak) -- the job of a simulation program.  "lattice" and
            "precision" choose the update: the SSLBM storages, the D2Q9 lattice, the varying
            diffusivity, the two-pass SLBM.
  bgk       the same with the BGK comparison scheme.
  fd4       the same with the finite-difference RK4 reference (order 4 or 2).
  ensemble  many scenarios of uneven size in one handle: write all, run, totals, read all.
  infer     the learned surrogate: network input from the states, one inference.
  train     one surrogate training step (forward, loss, backward, optimizer), gradients read.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2603_19789_gb300 import inputs
from paper_2603_19789_gb300 import sslbm as L
from paper_2603_19789_gb300 import surrogate

LATTICES = {"d2q5": L.LATTICE_D2Q5, "d2q9": L.LATTICE_D2Q9, "slbm": L.LATTICE_D2Q5_SLBM, "vard": L.LATTICE_D2Q5_VARD}
BCS = {"periodic": L.BC_PERIODIC, "noflux": L.BC_NOFLUX}


def _grid(name, nx, ny, steps, bc="periodic", precision="fp32", lattice="d2q5", units="lattice", diag=False,
          tune=False):
    return {"name": name, "kind": "grid", "nx": nx, "ny": ny, "steps": steps, "bc": bc, "precision": precision,
            "lattice": lattice, "units": units, "diag": diag, "tune": tune}


def listed():
    return [
        # the README's and the parity workload's grid: a small interactive run, where launch
        # latency counts
        _grid("sslbm_fp32_128", 128, 128, 200),
        # the paper's test case (Sec. III): 200 x 200 km in physical units, double precision
        _grid("sslbm_fp64_200", 200, 200, 100, precision="fp64", units="paper"),
        # an ordinary simulation domain of odd, ragged size with walls, monitored by its totals
        _grid("sslbm_fp32_1001x777", 1001, 777, 100, bc="noflux", diag=True),
        # the benchmark's grid: the largest production run, with the blocking tuned for it
        _grid("sslbm_fp32_8192", 8192, 8192, 100, bc="noflux", diag=True, tune=True),
        # a run that needs double accuracy at speed (the double-word storage)
        _grid("sslbm_fp64dw_1024", 1024, 1024, 50, bc="noflux", precision="fp64_dw"),
        # the isotropic lattice, walls, a width that is no multiple of the strips
        _grid("d2q9_fp32_1500x1100", 1500, 1100, 60, bc="noflux", lattice="d2q9"),
        # mobility map: spatially varying, anisotropic diffusivity
        _grid("vard_fp32_2048", 2048, 2048, 40, bc="noflux", lattice="vard"),
        # the paper's comparison scheme
        {"name": "bgk_fp32_2048", "kind": "bgk", "nx": 2048, "ny": 2048, "steps": 20, "bc": "periodic",
         "precision": "fp32"},
        # the finite-difference reference that the accuracy and cost studies run
        {"name": "fd4_fp32_1000", "kind": "fd4", "nx": 1000, "ny": 1000, "steps": 20, "bc": "periodic",
         "precision": "fp32", "order": 4},
        # a scenario sweep (parameter study) of uneven grid sizes
        {"name": "ensemble_fp32_32", "kind": "ensemble", "scenarios": 32, "max_size": 1024, "steps": 200,
         "precision": "fp32"},
        # surrogate serving: a batch of scenarios advanced by one network evaluation
        {"name": "surrogate_infer_64x256", "kind": "infer", "n": 256, "batch": 64, "width": 32, "modes": 12,
         "layers": 4, "hidden": 64},
        # surrogate training at the study's batch size
        {"name": "surrogate_train_16x256", "kind": "train", "n": 256, "batch": 16, "width": 32, "modes": 12,
         "layers": 4, "hidden": 64},
    ]


# Cell-steps of a drawn grid case, by update: about the time of the largest listed case.
_CAP = {("d2q5", "fp32"): 4e9, ("d2q5", "fp32_dev"): 4e9, ("d2q5", "fp32_split"): 3e9, ("d2q5", "fp32_kahan"): 1.2e9,
        ("d2q5", "fp64_dw"): 3e8, ("d2q5", "fp64"): 1e8, ("d2q9", "fp32"): 2e9, ("d2q9", "fp64"): 7e7,
        ("vard", "fp32"): 1.5e9, ("vard", "fp64"): 6e7, ("slbm", "fp32"): 6e8, ("slbm", "fp64"): 6e7,
        ("bgk", "fp32"): 4e8, ("bgk", "fp64"): 8e7, ("fd4", "fp32"): 1.4e8, ("fd4", "fp64"): 1e7}


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_size(rng, cap, max_steps=200):
    """nx, ny in [48, 4096] and steps in [1, max_steps], all over their logarithm, within cap cell-steps."""
    while True:
        nx, ny, steps = _log_int(rng, 48, 4096), _log_int(rng, 48, 4096), _log_int(rng, 1, max_steps)
        if rng.random() < 0.5:
            nx = max(48, nx // 4 * 4)
        if nx * ny * steps <= cap:
            return nx, ny, steps


def draw(rng):
    kind = rng.choices(["grid", "bgk", "fd4", "ensemble", "infer", "train"], [10, 2, 2, 2, 2, 2])[0]
    if kind in ("infer", "train"):
        width, modes, hidden = rng.choice([(32, 12, 64), (32, 12, 64), (16, 8, 32)])
        n = rng.choice([64, 128, 256])
        return {"kind": kind, "n": n, "batch": _log_int(rng, 1, 64 if kind == "infer" else 16), "width": width,
                "modes": modes, "layers": rng.choice([2, 3, 4]), "hidden": hidden}
    if kind == "ensemble":
        return {"kind": kind, "scenarios": _log_int(rng, 2, 48), "max_size": rng.choice([256, 512, 1024]),
                "steps": _log_int(rng, 4, 200), "precision": rng.choice(["fp32", "fp32", "fp32_dev", "fp32_split"])}
    bc = rng.choice(["periodic", "noflux"])
    if kind in ("bgk", "fd4"):
        precision = rng.choice(["fp32", "fp32", "fp64"])
        nx, ny, steps = _draw_size(rng, _CAP[kind, precision])
        case = {"kind": kind, "nx": nx, "ny": ny, "steps": steps, "bc": bc, "precision": precision}
        if kind == "fd4":
            case["order"] = rng.choice([4, 4, 2])
        return case
    lattice = rng.choice(["d2q5", "d2q5", "d2q5", "d2q9", "vard", "slbm"])
    if lattice == "d2q5":
        precision = rng.choice(["fp32", "fp32", "fp32", "fp32_dev", "fp32_split", "fp32_kahan", "fp64_dw", "fp64"])
    else:
        precision = rng.choice(["fp32", "fp32", "fp64"])
    nx, ny, steps = _draw_size(rng, _CAP[lattice, precision], 100 if precision == "fp64_dw" else 200)
    units = rng.choice(["lattice", "lattice", "paper"])
    case = _grid(None, nx, ny, steps, bc, precision, lattice, units, rng.random() < 0.3, False)
    del case["name"]
    return case


# ---------------------------------------------------------------------------
# inputs: the seeded infected Gaussians of the package's workloads, laid out on the GPU
# ---------------------------------------------------------------------------

def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _uniform(g, lo, hi, n):
    return torch.rand(n, generator=g, dtype=torch.float64) * (hi - lo) + lo


def _bumps(nx, ny, g, count, amp, periodic, width=1.0):
    """Sum of `count` Gaussians (amplitude U[amp], sigma U[4, 32] cells times width) at uniform
    positions, (ny, nx) float64: each is a product of a column and a row factor."""
    a = _uniform(g, amp[0], amp[1], count)
    sig = _uniform(g, 4.0, 32.0, count) * width
    cx, cy = _uniform(g, 0.0, nx, count), _uniform(g, 0.0, ny, count)

    def factor(n, c):
        d = torch.arange(n, dtype=torch.float64)[None, :] - c[:, None]
        if periodic:
            d = d - n * torch.round(d / n)
        f = torch.exp(-d * d / (2.0 * sig[:, None] ** 2))
        return torch.where(d.abs() <= 8.0 * sig[:, None], f, torch.zeros_like(f)).to(_dev())

    return (factor(ny, cy) * a.to(_dev())[:, None]).t() @ factor(nx, cx)


def _state(nx, ny, g, periodic, units):
    """Initial S, E, I, R, D, float64 (5, ny, nx) on the GPU."""
    st = torch.zeros((5, ny, nx), dtype=torch.float64, device=_dev())
    if units == "paper":  # E = chi N/A + eps, S the rest; 5e6 people on 200 x 200 cells
        dens = 125.0
        st[1] = 0.1 * dens * (1.0 + 2e-3 * (_noise(nx, ny, g) - 0.5))
        st[0] = dens - st[1]
        return st
    count = max(1, min(64, nx * ny // 16384))
    st[2] = _bumps(nx, ny, g, count, (1e-4, 1e-2), periodic) + 1e-6 * _noise(nx, ny, g)
    st[0] = 1.0 - st[2]
    return st


def _noise(nx, ny, g):
    dg = torch.Generator(device=_dev())
    dg.manual_seed(int(torch.randint(0, 2 ** 40, (1,), generator=g)))
    return torch.rand((ny, nx), generator=dg, dtype=torch.float64, device=_dev())


def _gen(seed):
    g = torch.Generator()
    g.manual_seed(int(seed))
    return g


def _params(case):
    """rates, d, dx, dt of a grid case: the package's workloads."""
    if case.get("units") == "paper":  # per day and km^2/day, dt = 0.01 day
        gamma = 1.0 / 5.0
        return dict(rates=(3.0 * gamma, 1.0 / 7.0, gamma, 0.3), d=(4.35e-2, 4.35e-2, 1e-4, 4.35e-2, 0.0), dx=1.0, dt=0.01)
    r = inputs.rates_from_sigma_mu(0.5, 0.2, 0.1, 0.01)
    return dict(rates=r.as_tuple(), d=(0.05, 0.05, 0.01, 0.05, 0.0), dx=1.0, dt=1.0)


def _grid_inputs(case, seed):
    g = _gen(seed)
    u = _state(case["nx"], case["ny"], g, case["bc"] == "periodic", case.get("units", "lattice"))
    kappa = None
    if case.get("lattice") == "vard":
        kx = 0.5 + 1.2 * torch.clamp(_bumps(case["nx"], case["ny"], g, 5, (0.5, 1.0), False, 4.0), max=1.0)
        kappa = (kx, kx * float(_uniform(g, 0.5, 1.0, 1)))
    if case["precision"] == "fp32":
        u = u.float()
        kappa = None if kappa is None else (kappa[0].float(), kappa[1].float())
    return u, kappa


def _surrogate_inputs(case, seed):
    """States in mid-epidemic, scenario parameters of the ensemble workload, network parameters,
    and (training) the states some steps later."""
    g = _gen(seed)
    n, batch = case["n"], case["batch"]
    u = torch.zeros((batch, 5, n, n), dtype=torch.float32, device=_dev())
    target = torch.zeros_like(u)
    for b in range(batch):
        count = int(torch.randint(1, 9, (1,), generator=g))
        pos = int(torch.randint(0, 2 ** 40, (1,), generator=g))
        amp = float(10.0 ** _uniform(g, -3.0, -1.3, 1))
        for t, (dst, w) in enumerate(((u, 1.0), (target, 1.1))):
            infected = _bumps(n, n, _gen(pos), count, (0.5 * amp, amp), True, w)
            removed = _bumps(n, n, _gen(pos), count, (0.5 * amp, amp), True, 0.7 * w)
            st = [None, 0.7 * infected, infected, 0.9 * (t + 1) * removed, 0.1 * (t + 1) * removed]
            st[0] = 1.0 - (st[1] + st[2] + st[3] + st[4])
            dst[b] = torch.stack(st).float()
    r0 = _uniform(g, 1.2, 4.0, batch).float().to(_dev())
    logd = _uniform(g, -3.0, -1.0, batch).float().to(_dev())
    theta = surrogate.initial_params(case["width"], case["modes"], case["layers"], case["hidden"], seed=seed % 2 ** 31)
    return u, target, r0, logd, theta


def _ensemble_inputs(case, seed):
    sizes = tuple(s for s in inputs.ENSEMBLE_SIZES if s <= case["max_size"])
    # the sizes are the case's, the parameters and states the seed's
    layout = inputs.ensemble_scenarios(case["scenarios"], sizes=sizes)
    sc = inputs.ensemble_scenarios(case["scenarios"], seed=seed, sizes=sizes)
    specs = [dict(nx=a["nx"], ny=a["ny"], rates=s["rates"].as_tuple(), d=s["d"]) for a, s in zip(layout, sc)]
    g = _gen(seed)
    states = [_state(sp["nx"], sp["ny"], g, True, "lattice").float() for sp in specs]
    return specs, states


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        specs, states = _ensemble_inputs(case, seed)
        ens = L.Ensemble(specs, precision=L.PRECISIONS[case["precision"]])
        return {"case": case, "ens": ens, "in": states, "out": [torch.empty_like(s) for s in states]}
    if kind in ("infer", "train"):
        u, target, r0, logd, theta = _surrogate_inputs(case, seed)
        sur = L.Surrogate(case["n"], case["width"], case["modes"], case["layers"], case["hidden"], case["batch"])
        sur.set_params(theta)
        st = {"case": case, "sur": sur, "u": u, "r0": r0, "logd": logd}
        if kind == "train":
            sur.set_loss_weights(0.0, 30.0)
            st["target"] = target
            st["grads"] = torch.empty(sur.nparams, dtype=torch.float32, device=_dev())
        return st
    u, kappa = _grid_inputs(case, seed)
    p = _params(case)
    precision = L.PRECISIONS[case["precision"]]
    if kind == "fd4":
        s = L.Fd4(case["nx"], case["ny"], p["rates"], p["d"], p["dx"], _fd4_dt(p), BCS[case["bc"]], precision,
                  case["order"])
    elif kind == "bgk":
        s = L.Solver(case["nx"], case["ny"], p["rates"], d=p["d"], dx=p["dx"], dt=p["dt"], bc=BCS[case["bc"]],
                     precision=precision, schemes=L.WANT_BGK)
    else:
        s = L.Solver(case["nx"], case["ny"], p["rates"], d=p["d"], dx=p["dx"], dt=p["dt"], bc=BCS[case["bc"]],
                     precision=precision, lattice=LATTICES[case["lattice"]],
                     s_ref=125.0 if case["units"] == "paper" else 1.0)
        if kappa is not None:
            s.set_diffusivity_scale(*kappa)
        if case["tune"]:
            s.write(u)
            s.autotune()
    return {"case": case, "solver": s, "in": u, "out": torch.empty_like(u)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "ensemble":
        ens = state["ens"]
        for i, u in enumerate(state["in"]):
            ens.write(i, u)
        ens.run(case["steps"])
        totals, peak = ens.diagnostics()
        for i, out in enumerate(state["out"]):
            L.sslbm_ensemble_read(ens.e, i, out)
        return {"states": state["out"], "totals": totals, "peak": peak}
    if kind == "infer":
        sur = state["sur"]
        x = sur.make_input(state["u"], state["r0"], state["logd"])
        return {"x": x, "y": sur.infer(x)}
    if kind == "train":
        # the first step of a warm-up schedule: learning rate 0, so that every pass takes the
        # gradients at the same parameters
        sur = state["sur"]
        x = sur.make_input(state["u"], state["r0"], state["logd"])
        loss = sur.train_step(x, state["target"], 0.0)
        return {"loss": loss, "grads": L.sslbm_fno_get_grads(sur.f, state["grads"])}
    s = state["solver"]
    if kind == "fd4":
        s.write(state["in"])
        s.step(case["steps"])
        return {"state": L.sslbm_fd4_read(s.f, state["out"])}
    scheme = L.SCHEME_BGK if kind == "bgk" else L.SCHEME_SSLBM
    s.write(state["in"], scheme=scheme)
    if kind == "bgk":
        s.bgk_step(case["steps"])
        return {"state": L.sslbm_read(s.h, scheme, L.ALL, state["out"])}
    s.step(case["steps"])
    res = {}
    if case["diag"]:
        res["totals"], res["peak"] = s.diagnostics()
    res["state"] = L.sslbm_read(s.h, scheme, L.ALL, state["out"])
    return res


def _fd4_dt(p):
    return p["dt"] * 0.25  # the accuracy study's step: a quarter of the SSLBM's


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------

# floating-point operations per cell and step of each update, divisions counted once
_FLOPS = {"d2q5": 46, "d2q9": 66, "vard": 82, "slbm": 70, "bgk": 170, "fd4": 460}


def work(case):
    kind = case["kind"]
    if kind == "ensemble":
        sizes = tuple(s for s in inputs.ENSEMBLE_SIZES if s <= case["max_size"])
        cells = sum(s["nx"] * s["ny"] for s in inputs.ensemble_scenarios(case["scenarios"], sizes=sizes))
        return {"bytes": 2 * 20 * cells, "flops": _FLOPS["d2q5"] * cells * case["steps"]}
    if kind in ("infer", "train"):
        n, b = case["n"], case["batch"]
        shape = (n, case["width"], case["modes"], case["layers"], case["hidden"])
        fwd = surrogate.forward_flops(*shape)
        params = 4 * len_params(case)
        if kind == "infer":  # states in, network input and prediction out
            return {"bytes": b * n * n * 4 * (5 + 8 + 5) + params, "flops": b * fwd}
        # states and targets in; parameters, gradients and the two moments read and written
        return {"bytes": b * n * n * 4 * (5 + 5) + 7 * params, "flops": 3 * b * fwd}
    cells = case["nx"] * case["ny"]
    size = 4 if case["precision"] == "fp32" else 8
    planes = 10 + (2 if case.get("lattice") == "vard" else 0)
    key = case["lattice"] if kind == "grid" else kind
    return {"bytes": planes * size * cells, "flops": _FLOPS[key] * cells * case["steps"]}


def len_params(case):
    W, m, H = case["width"], case["modes"], case["hidden"]
    return 9 * W + case["layers"] * (W * W * 2 * m * m * 2 + W * W + W) + H * W + H + 5 * H + 5


# ---------------------------------------------------------------------------
# exact: the same outputs from plain torch in 64 bits
# ---------------------------------------------------------------------------

def _shift(f, dx, dy, bc):
    """f(x + dx, y + dy) on the last two axes; beyond a no-flux wall the nearest cell's mirror image."""
    ny, nx = f.shape[-2:]
    if bc == "periodic":
        return torch.roll(f, (-dy, -dx), (-2, -1))
    if dx:
        i = torch.arange(nx, device=f.device) + dx
        i = torch.where(i < 0, -1 - i, torch.where(i >= nx, 2 * nx - 1 - i, i))
        f = f.index_select(-1, i)
    if dy:
        i = torch.arange(ny, device=f.device) + dy
        i = torch.where(i < 0, -1 - i, torch.where(i >= ny, 2 * ny - 1 - i, i))
        f = f.index_select(-2, i)
    return f


def _link(f, dx, dy, bc):
    """f(x + dx, y + dy), or the cell's own value where that link leaves a no-flux domain."""
    s = _shift(f, dx, dy, bc)
    if bc == "periodic" or not (dx and dy):
        return s
    ny, nx = f.shape[-2:]
    edge = torch.zeros((ny, nx), dtype=torch.bool, device=f.device)
    edge[:, nx - 1 if dx > 0 else 0] = True
    edge[ny - 1 if dy > 0 else 0, :] = True
    return torch.where(edge, f, s)


def _lap5(f, bc):
    return _shift(f, 1, 0, bc) + _shift(f, -1, 0, bc) + _shift(f, 0, 1, bc) + _shift(f, 0, -1, bc) - 4.0 * f


def _lap9(f, bc):
    axes = sum(_link(f, dx, dy, bc) for dx, dy in ((1, 0), (-1, 0), (0, 1), (0, -1)))
    diag = sum(_link(f, dx, dy, bc) for dx, dy in ((1, 1), (-1, 1), (1, -1), (-1, -1)))
    return (4.0 * axes + diag - 20.0 * f) / 6.0


def _force(S, E, I, R, beta):
    n = S + E + I + R
    return torch.where(n > 0, beta * S * I / torch.where(n > 0, n, torch.ones_like(n)), torch.zeros_like(n))


def _rates(p):
    beta, alpha, gamma, phi = p["rates"]
    return beta * p["dt"], alpha * p["dt"], (1.0 - phi) * gamma * p["dt"], phi * gamma * p["dt"]


def _sources(u, p):
    """Psi dt of the five compartments."""
    bdt, adt, rdt, ddt = _rates(p)
    S, E, I, R = u[0], u[1], u[2], u[3]
    F = _force(S, E, I, R, bdt)
    return torch.stack([-F, F - adt * E, adt * E - (rdt + ddt) * I, rdt * I, ddt * I])


def _exact_grid(case, u, kappa, p):
    bc, lattice = case["bc"], case.get("lattice", "d2q5")
    d = [p["d"][c] * p["dt"] / p["dx"] ** 2 for c in range(4)]
    if kappa is not None:
        kx, ky = kappa
        links = [(dx, dy, 0.5 * (k + _shift(k, dx, dy, bc)))
                 for dx, dy, k in ((1, 0, kx), (-1, 0, kx), (0, 1, ky), (0, -1, ky))]
    for _ in range(case["steps"]):
        n = _sources(u, p)
        for c in range(4):
            f = u[c]
            if lattice == "vard":
                n[c] += d[c] * sum(k * (_shift(f, dx, dy, bc) - f) for dx, dy, k in links) + f
            elif lattice == "slbm":
                ps = f + _lap5(f, bc) / 6.0
                n[c] += ps + (3.0 * d[c] - 0.5) * (ps + _lap5(ps, bc) / 6.0 - f)
            else:
                n[c] += f + d[c] * (_lap9(f, bc) if lattice == "d2q9" else _lap5(f, bc))
        n[4] += u[4]
        u = n
    return u


def _exact_bgk(case, u, p):
    bc = case["bc"]
    tau = torch.tensor([3.0 * p["d"][c] * p["dt"] / p["dx"] ** 2 + 0.5 for c in range(4)], dtype=torch.float64,
                       device=u.device)[:, None, None]
    w = (1 / 3, 1 / 6, 1 / 6, 1 / 6, 1 / 6)
    c = ((0, 0), (1, 0), (0, 1), (-1, 0), (0, -1))
    f = [wi * u[:4] for wi in w]
    D = u[4]
    for _ in range(case["steps"]):
        rho = sum(f)
        psi = _sources(rho, p)
        post = [f[i] + (w[i] * rho - f[i]) / tau + w[i] * psi[:4] for i in range(5)]
        D = D + psi[4]
        new = []
        for i, (cx, cy) in enumerate(c):  # pull: f_i(x) = post_i(x - c_i), at a wall the opposite population
            s = torch.roll(post[i], (cy, cx), (-2, -1))
            if bc == "noflux" and i:
                opp = post[(0, 3, 4, 1, 2)[i]]
                if cx:
                    j = 0 if cx > 0 else s.shape[-1] - 1
                    s[..., j] = opp[..., j]
                else:
                    j = 0 if cy > 0 else s.shape[-2] - 1
                    s[..., j, :] = opp[..., j, :]
            new.append(s)
        f = new
    return torch.cat([sum(f), D[None]])


def _exact_fd4(case, u, p):
    bc, dt = case["bc"], _fd4_dt(p)
    unit = dict(p, dt=1.0)

    def axis(f, dx, dy):
        near = _shift(f, dx, dy, bc) + _shift(f, -dx, -dy, bc)
        if case["order"] == 2:
            return (near - 2.0 * f) / p["dx"] ** 2
        far = _shift(f, 2 * dx, 2 * dy, bc) + _shift(f, -2 * dx, -2 * dy, bc)
        return (16.0 * near - far - 30.0 * f) / (12.0 * p["dx"] ** 2)

    def rhs(v):
        r = _sources(v, unit)
        for c in range(4):
            r[c] += p["d"][c] * (axis(v[c], 1, 0) + axis(v[c], 0, 1))
        return r

    for _ in range(case["steps"]):
        k1 = rhs(u)
        k2 = rhs(u + 0.5 * dt * k1)
        k3 = rhs(u + 0.5 * dt * k2)
        k4 = rhs(u + dt * k3)
        u = u + dt / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
    return u


def _gelu(z):
    return 0.5 * z * (1.0 + torch.tanh(math.sqrt(2.0 / math.pi) * (z + 0.044715 * z ** 3)))


def _exact_net(case, u, r0, logd, theta):
    """Network input and prediction of a batch, differentiable in theta (float64)."""
    W, m, H, n = case["width"], case["modes"], case["hidden"], case["n"]
    off = 0

    def take(*shape):
        nonlocal off
        size = int(np.prod(shape))
        off += size
        return theta[off - size:off].reshape(shape)

    s = torch.clamp(u[:, 1:3].amax(dim=(1, 2, 3)), min=1e-12)
    e = (torch.log10(s) + 4.0) / 4.0
    sp = 10.0 ** (4.0 * e - 4.0)
    sig = torch.ones((u.shape[0], 5), dtype=torch.float64, device=u.device)
    sig[:, 1] = sp
    sig[:, 2] = sp
    sig = sig[:, :, None, None]
    const = torch.stack([(r0 - 2.6) / 1.4, logd + 2.0, e], dim=1)[:, :, None, None].expand(-1, -1, n, n)
    x = torch.cat([u / sig, const], dim=1)
    kx = torch.tensor([j if j < m else n - 2 * m + j for j in range(2 * m)], device=u.device)
    cw = torch.full((m, 1), 2.0, dtype=torch.float64, device=u.device)
    cw[0] = 1.0
    A0, a0 = take(W, 8), take(W)
    h = torch.einsum("oi,biyx->boyx", A0, x) + a0[:, None, None]
    for layer in range(case["layers"]):
        R = torch.view_as_complex(take(W, W, 2 * m, m, 2).contiguous())
        Bl, bl = take(W, W), take(W)
        hat = torch.fft.fft2(h)[:, :, :m][..., kx]                     # [b, i, ky, kx]
        g = torch.einsum("biqk,iokq->boqk", hat, R) * cw
        G = torch.zeros((u.shape[0], W, n, n), dtype=torch.complex128, device=u.device)
        G = G.index_put((torch.arange(u.shape[0], device=u.device)[:, None, None, None],
                         torch.arange(W, device=u.device)[:, None, None],
                         torch.arange(m, device=u.device)[:, None], kx), g)
        z = torch.fft.ifft2(G).real + torch.einsum("oi,biyx->boyx", Bl, h) + bl[:, None, None]
        h = _gelu(z) if layer < case["layers"] - 1 else z
    Q1, q1, Q2, q2 = take(H, W), take(H), take(5, H), take(5)
    q = _gelu(torch.einsum("oi,biyx->boyx", Q1, h) + q1[:, None, None])
    delta = torch.einsum("oi,biyx->boyx", Q2, q) + q2[:, None, None]
    v = sig * torch.clamp(x[:, :5] + delta, min=0.0)
    su, sv = (sig * x[:, :5]).sum(dim=(1, 2, 3)), v.sum(dim=(1, 2, 3))
    y = v * (su / torch.clamp(sv, min=1e-300))[:, None, None, None]
    return x, y, sig


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        specs, states = _ensemble_inputs(case, seed)
        outs = []
        for sp, u in zip(specs, states):
            p = dict(rates=sp["rates"], d=sp["d"], dx=1.0, dt=1.0)
            outs.append(_exact_grid({"bc": "periodic", "steps": case["steps"]}, u.double(), None, p))
        totals = np.stack([o.sum(dim=(1, 2)).cpu().numpy() for o in outs])
        return {"states": outs, "totals": totals, "peak": np.array([float(o[2].max()) for o in outs])}
    if kind in ("infer", "train"):
        u, target, r0, logd, theta = _surrogate_inputs(case, seed)
        th = torch.from_numpy(theta).double().to(_dev())
        u, target, r0, logd = u.double(), target.double(), r0.double(), logd.double()
        if kind == "infer":
            with torch.no_grad():
                parts = [_exact_net(case, u[b:b + 4], r0[b:b + 4], logd[b:b + 4], th)
                         for b in range(0, case["batch"], 4)]
            return {"x": torch.cat([q[0] for q in parts]), "y": torch.cat([q[1] for q in parts])}
        th.requires_grad_(True)
        loss = 0.0
        for b in range(0, case["batch"], 2):
            _, y, sig = _exact_net(case, u[b:b + 2], r0[b:b + 2], logd[b:b + 2], th)
            part = (((y - target[b:b + 2]) / sig) ** 2).sum() / target.numel()
            part.backward()
            loss += float(part.detach())
        return {"loss": loss, "grads": th.grad}
    u, kappa = _grid_inputs(case, seed)
    u = u.double()
    kappa = None if kappa is None else tuple(k.double() for k in kappa)
    p = _params(case)
    if kind == "fd4":
        return {"state": _exact_fd4(case, u, p)}
    if kind == "bgk":
        return {"state": _exact_bgk(case, u, p)}
    out = _exact_grid(case, u, kappa, p)
    res = {}
    if case["diag"]:
        res["totals"], res["peak"] = out.sum(dim=(1, 2)).cpu().numpy(), float(out[2].max())
    res["state"] = out
    return res
