"""Timed cases of the library: what a program that uses it has it do, one pass each.

A case is a dict of plain values. Its "kind" says which of the public classes carries it:

  run      one lattice (lbm.Lattice): a chunk of time steps, the GPU diagnostic that a run of
           that sort reads between chunks, and the populations as a checkpoint in page-locked
           host memory
  batch    many lattices (lbm.Batch): chunks of 64 steps, each followed by the Laplace
           measurement of every lattice, and the populations of one of them
  train    the surrogate network (lbm.MLP): full-batch Adam steps on the resident samples
  choose   the surrogate network: predictions for given points and kappa for given targets

prepare() makes the state a program holds before the pass, run() is the pass, work() counts
what it cannot do without, and exact() computes the same outputs in 64 bits with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1306_6445_gb300 import inputs, lbm

G = -1.0
SIGMA_F = 0.087        # Eq. 8 of the batched sweeps and of the Eq. 23 fluid
RHO_1 = 1.49           # density below which the splash relaxes at the vapour viscosity


def listed():
    return [
        # the FP64 validation run: one 128 x 128 droplet of radius 30, Laplace reading per chunk
        {"name": "fp64_droplet_128", "kind": "run", "prec": "fp64", "nx": 128, "ny": 128,
         "state": "droplet", "kappa": 0.5, "t": 0.8, "steps": 100, "read": "droplet",
         "tune": False, "resume": False},
        # an FP64 reference run of ragged size continued from a checkpoint
        {"name": "fp64_resume_1000x700", "kind": "run", "prec": "fp64", "nx": 1000, "ny": 700,
         "state": "droplet", "kappa": 0.3, "t": 0.8, "steps": 20, "read": "none",
         "tune": True, "resume": True},
        # the smallest lattice of the sweeps, run by itself with the mass and |v| of a log line
        {"name": "fp32_droplet_64", "kind": "run", "prec": "fp32", "nx": 64, "ny": 64,
         "state": "droplet", "kappa": 0.3, "t": 0.8, "steps": 50, "read": "reduce",
         "tune": False, "resume": False},
        # a logged run of an ordinary, odd-sized lattice as a program makes it (no autotuning)
        {"name": "fp32_droplet_501x383", "kind": "run", "prec": "fp32", "nx": 501, "ny": 383,
         "state": "droplet", "kappa": 0.6, "t": 0.8, "steps": 200, "read": "droplet",
         "tune": False, "resume": False},
        # the benchmark's droplet: 2048 x 2048, 100 steps and one reduction
        {"name": "fp32_droplet_2048", "kind": "run", "prec": "fp32", "nx": 2048, "ny": 2048,
         "state": "droplet", "kappa": 0.6, "t": 0.8, "steps": 100, "read": "reduce",
         "tune": True, "resume": False},
        # the capillary wave between walls, its interface read after each chunk
        {"name": "fp32_wave_4096x2048", "kind": "run", "prec": "fp32", "nx": 4096, "ny": 2048,
         "state": "layer", "kappa": 0.5, "t": 0.8, "steps": 100, "read": "height",
         "tune": True, "resume": False},
        # the benchmark's droplet in BF16 storage with the rounding that keeps its physics
        {"name": "bf16_droplet_2048", "kind": "run", "prec": "bf16", "nx": 2048, "ny": 2048,
         "state": "droplet", "kappa": 0.0, "t": 0.8, "steps": 100, "read": "reduce",
         "tune": True, "resume": False},
        # the droplet splash from its start to the first time of the spread-radius table
        {"name": "fp32_splash_600x225", "kind": "run", "prec": "fp32", "nx": 600, "ny": 225,
         "state": "splash", "kappa": 0.0, "t": 0.8, "steps": 160, "read": "none",
         "tune": False, "resume": False},
        # the sweep over 512 droplets of 64..512: one tick of its reading window
        {"name": "sweep_512_lattices", "kind": "batch", "n": 512, "side": 0, "sweep": 1306,
         "ticks": 1, "tune": True},
        # a Laplace check of chosen kappas: 24 lattices of 128 x 128, eight readings
        {"name": "laplace_check_24x128", "kind": "batch", "n": 24, "side": 128, "sweep": 7,
         "ticks": 8, "tune": True},
        # the surrogate's training on the sweep's 512 results
        {"name": "surrogate_train_512", "kind": "train", "n": 512, "steps": 50},
        # the surrogate's use: predictions and kappa for a table of targets
        {"name": "surrogate_choose_4097", "kind": "choose", "n": 4097},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above: any size between the smallest and the largest, odd
    ones among them, every storage type, boundary and diagnostic."""
    pick = rng.random()
    if pick < 0.66:
        prec = rng.choice(["fp32", "fp32", "fp32", "fp64", "bf16"])
        state = rng.choice(["droplet", "droplet", "layer", "splash"])
        if state == "splash" and prec == "bf16":     # not compiled for open boundaries
            state = "droplet"
        most = 1 << (20 if prec == "fp64" else 23)
        if state == "splash":
            s = math.exp(rng.uniform(0.0, math.log(3.0 if prec == "fp32" else 1.5)))
            nx, ny = int(600 * s) + rng.randint(0, 3), int(225 * s) + rng.randint(0, 3)
            steps, read = 160, rng.choice(["none", "reduce"])
        else:
            nx = _log_int(rng, 64, 4096)
            ny = _log_int(rng, 64, 2048)
            while nx * ny > most or max(nx, ny) > 4 * min(nx, ny):
                nx, ny = _log_int(rng, 64, 4096), _log_int(rng, 64, 2048)
            steps = int((4e7 if prec == "fp64" else 4e8) / (nx * ny))
            steps = max(20, min(200, steps)) - rng.randint(0, 1)
            read = rng.choice(["none", "reduce", "height" if state == "layer" else "droplet"])
        return {"kind": "run", "prec": prec, "nx": nx, "ny": ny, "state": state,
                "kappa": round(rng.uniform(0.0, 0.7), 3), "t": round(rng.uniform(0.8, 0.88), 3),
                "steps": steps, "read": read, "tune": rng.random() < 0.5,
                "resume": state != "splash" and rng.random() < 0.2}
    if pick < 0.83:
        side = rng.choice([0, 0, 32 * rng.randint(2, 10)])
        n = _log_int(rng, 6, 400 if side == 0 else min(512, max(8, int(2e7 / side**2))))
        sites = n * (side or 320) ** 2
        return {"kind": "batch", "n": n, "side": side, "sweep": rng.randint(1, 10**6),
                "ticks": rng.randint(1, max(1, min(8, int(4e7 / sites)))),
                "tune": rng.random() < 0.7}
    if pick < 0.92:
        return {"kind": "train", "n": _log_int(rng, 100, 6000), "steps": 50}
    return {"kind": "choose", "n": _log_int(rng, 24, 60000)}


# --------------------------------------------------------------------------------------
# set-up
# --------------------------------------------------------------------------------------

def _grid(nx, ny):
    y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
    x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :]
    return y, x


def _maxwell(t):
    eos = lbm.cs_eos(t)
    rv, rl, _ = lbm.lb_maxwell(eos, G)
    return eos, rv, rl


def _droplet(nx, ny, cx, cy, r, rl, rv):
    y, x = _grid(nx, ny)
    d = torch.sqrt((x - cx) ** 2 + (y - cy) ** 2)
    return 0.5 * (rl + rv) - 0.5 * (rl - rv) * torch.tanh(d - r)


def _splash_scale(case):
    return case["ny"] / 225.0


def _fields(case, seed):
    """Initial density and velocity ([ny][nx], float64, device) and the nominal radius: the
    droplet sits within a site or two of the centre, the layer's wave has a phase of its own,
    and a faint smooth flow (a few 1e-4) tells one seed's inputs from another's."""
    rng = np.random.default_rng(seed)
    nx, ny = case["nx"], case["ny"]
    y, x = _grid(nx, ny)
    radius = 0.0
    if case["state"] == "splash":
        s = _splash_scale(case)
        d, film, u = 100.0 * s, 25.0 * s, 0.125
        cx, cy = 0.5 * nx + rng.uniform(-2, 2), film + 0.5 * d - 0.05 * d
        f_film = 0.5 * (1 - torch.tanh(y + 0.5 - film)) * torch.ones_like(x)
        f_drop = 0.5 * (1 - torch.tanh(torch.sqrt((x - cx) ** 2 + (y - cy) ** 2) - 0.5 * d))
        rho = 1.0 + 99.0 * torch.maximum(f_film, f_drop)
        return rho, torch.zeros_like(rho), -u * f_drop, 0.5 * d
    _, rv, rl = _maxwell(case["t"])
    if case["state"] == "droplet":
        radius = 0.234375 * min(nx, ny)
        rho = _droplet(nx, ny, 0.5 * (nx - 1) + rng.uniform(-1.5, 1.5),
                       0.5 * (ny - 1) + rng.uniform(-1.5, 1.5),
                       radius * rng.uniform(0.98, 1.02), rl, rv)
    else:
        h = 0.5 * ny + 0.01 * nx * torch.cos(2 * math.pi * x / nx + rng.uniform(0, 2 * math.pi))
        rho = 0.5 * (rl + rv) - 0.5 * (rl - rv) * torch.tanh(y - h)
    a, p = rng.uniform(1e-4, 4e-4, 2), rng.uniform(0, 2 * math.pi, 2)
    ux = a[0] * torch.sin(2 * math.pi * y / ny + p[0]) * torch.ones_like(x)
    uy = a[1] * torch.sin(2 * math.pi * x / nx + p[1]) * torch.ones_like(y)
    if case["state"] == "layer":       # nothing flows through the walls at the start
        uy = uy * torch.sin(math.pi * (y + 0.5) / ny)
    return rho, ux, uy, radius


def _rates(case):
    if case["state"] == "splash":      # Re = 1000 at U = 0.125
        return lbm.RateParams.from_viscosity(0.125 * 100.0 * _splash_scale(case) / 1000.0)
    return lbm.RateParams.from_viscosity(0.1)


def _shift(case):
    return _maxwell(case["t"])[1] if case["prec"] == "bf16" else 0.0


def _prepare_run(case, seed):
    nx, ny, prec = case["nx"], case["ny"], case["prec"]
    rho, ux, uy, radius = _fields(case, seed)
    kw = {}
    if case["state"] == "splash":
        nu_v = 20.0 * 0.125 * 100.0 * _splash_scale(case) / 1000.0
        eos, sigma = lbm.EOSParams(kind="piecewise"), SIGMA_F
        kw = {"open_bc": True, "viscosity_switch": (RHO_1, 1.0 / (3.0 * nu_v + 0.5))}
    else:
        eos, sigma = lbm.cs_eos(case["t"]), 0.0
        kw = {"walls_y": case["state"] == "layer"}
    if prec == "bf16":
        kw.update(storage_shift=_shift(case), stochastic_rounding=True)
    lat = lbm.Lattice(nx, ny, eos, G, kappa=case["kappa"], sigma_force=sigma,
                      rates=_rates(case), prec=prec, **kw)
    host = [np.ascontiguousarray(v.cpu().numpy()) for v in (rho, ux, uy)]
    lat.set_rho_u(*host)
    if case["tune"]:
        lat.autotune()
    kind = {"fp64": torch.float64, "fp32": torch.float32, "bf16": torch.bfloat16}[prec]
    pops = torch.empty((9, ny, nx), dtype=kind, pin_memory=True)
    s = {"case": case, "lat": lat, "host": host, "radius": radius, "pops": pops, "saved": None,
         "mid": float(rho.max() + rho.min()) / 2}
    if case["resume"]:
        s["saved"] = torch.empty_like(pops, pin_memory=True)
        lbm.lb_get_populations(lat.ctx, s["saved"].data_ptr(), _nbytes(pops))
    return s


def _nbytes(t):
    return t.numel() * t.element_size()


def _run_run(s):
    case, lat = s["case"], s["lat"]
    if case["state"] == "splash":      # the run begins at the impact
        lat.set_rho_u(*s["host"])
    elif case["resume"]:
        lbm.lb_set_populations(lat.ctx, s["saved"].data_ptr(), _nbytes(s["saved"]))
    lat.step(case["steps"])
    out = {}
    # the readings of a run are logged in single precision
    if case["read"] == "reduce":
        out["sums"] = lat.reduce().astype(np.float32)
    elif case["read"] == "droplet":
        out["droplet"] = np.array(list(lat.measure_droplet(s["radius"]).values()), np.float32)
    elif case["read"] == "height":
        out["height"] = lat.interface_height(s["mid"]).astype(np.float32)
    lbm.lb_get_populations(lat.ctx, s["pops"].data_ptr(), _nbytes(s["pops"]))
    out["populations"] = s["pops"]
    return out


def _batch_rows(case):
    """The case's lattices: side, T/T_c, kappa, tau_v, nominal radius."""
    rows = []
    for d in inputs.batch_draws(case["n"], case["sweep"]):
        side = case["side"] or d["side"]
        radius = 0.25 * side if case["side"] else d["radius"]
        rows.append((side, d["t_over_tc"], d["kappa"], d["tau_v"], radius))
    return rows


def _batch_density(case, seed):
    """(rows, per-lattice initial density on the device)."""
    rng = np.random.default_rng(seed)
    rows = _batch_rows(case)
    rho = []
    for side, t, _, _, radius in rows:
        _, rv, rl = _maxwell(t)
        c = 0.5 * (side - 1)
        rho.append(_droplet(side, side, c + rng.uniform(-1, 1), c + rng.uniform(-1, 1),
                            radius * rng.uniform(0.98, 1.02), rl, rv))
    return rows, rho


def _prepare_batch(case, seed):
    rows, rho = _batch_density(case, seed)
    descs = [lbm.LatticeDesc(side, side, lbm.cs_eos(t), G, kappa=kappa, sigma_force=SIGMA_F,
                             rates=lbm.RateParams(s_v=1.0 / tau))
             for side, t, kappa, tau, _ in rows]
    b = lbm.Batch(descs, prec="fp32")
    for i, r in enumerate(rho):
        b.set_rho_u(i, r.cpu().numpy())
    if case["tune"]:
        b.autotune(2)
    return {"case": case, "batch": b, "radii": np.array([r[4] for r in rows])}


def _run_batch(s):
    b, readings = s["batch"], []
    for _ in range(s["case"]["ticks"]):
        b.step(64)
        readings.append(b.measure(s["radii"]))
    # the training data of the surrogate is kept in single precision
    return {"readings": np.asarray(readings, dtype=np.float32),
            "populations": b.populations(s["case"]["n"] // 2)}


# ---- the surrogate

def _samples(n, seed):
    """Training points over the sweep's ranges with results of the sweep's shape: sigma
    falls with kappa and as (1 - T)^1.5, the densities follow T."""
    rng = np.random.default_rng(seed)
    x = np.stack([rng.uniform(0.65, 0.95, n), rng.uniform(0, 0.95, n), rng.uniform(0.6, 1.2, n)],
                 axis=1)
    t, k, tau = x.T
    y = np.stack([0.06 * (1 - k) * (1 - t) ** 1.5 * (1 + 0.02 * (tau - 0.9)),
                  0.55 - 0.8 * (t - 0.65) ** 2, 0.002 + 0.3 * (t - 0.6) ** 2], axis=1)
    return x.astype(np.float32), y.astype(np.float32)


_LR = 1e-3


def _prepare_train(case, seed):
    x, y = _samples(case["n"], seed)
    net = lbm.MLP(case["n"])
    net.set_params(inputs.mlp_init(seed))
    net.set_data(x, y)
    return {"case": case, "net": net}


def _run_train(s):
    loss = s["net"].train(s["case"]["steps"], _LR)
    return {"loss": np.array([loss], np.float32), "params": s["net"].params()}


def _trained_like(seed):
    """Saved parameters of a network whose sigma falls with kappa, as a trained one's does
    (the kappa feature reaches the hidden layers with positive weights on GELU's increasing
    branch), and its normalisation."""
    rng = np.random.default_rng(seed)
    h = 64
    w1 = rng.uniform(-0.05, 0.05, (h, 3))
    w1[:, 1] = rng.uniform(0.02, 0.12, h)
    b1 = rng.uniform(0.8, 1.2, h)
    w2 = rng.uniform(0.0, 0.03, (h, h))
    b2 = rng.uniform(-0.1, 0.1, h)
    w3 = rng.uniform(-0.1, 0.1, (3, h))
    w3[0] = rng.uniform(0.05, 0.15, h)
    b3 = rng.uniform(-0.1, 0.1, 3) - np.array([4.0, 0.0, 0.0])
    theta = np.concatenate([v.ravel() for v in (w1, b1, w2, b2, w3, b3)]).astype(np.float32)
    norm = [np.array(v, np.float32) for v in
            ((-1.6, -0.9, 0.9), (0.5, 0.75, 0.17), (-6.5, 0.5, -3.6), (1.2, 0.06, 1.0))]
    return theta, norm


def _choose_inputs(case, seed):
    """(parameters, normalisation, points to predict, (T/T_c, tau_v, sigma) queries)."""
    theta, norm = _trained_like(seed)
    x, _ = _samples(case["n"], seed + 1)
    goal = np.clip(x, [0.0, 0.03, 0.0], [1.0, 0.92, 2.0]).astype(np.float32)
    sigma = _net(theta, norm, goal)[0][:, 0].cpu().numpy()
    return theta, norm, x, np.stack([goal[:, 0], goal[:, 2], sigma], axis=1).astype(np.float32)


def _prepare_choose(case, seed):
    theta, norm, x, queries = _choose_inputs(case, seed)
    net = lbm.MLP(1)
    net.set_params(theta)
    net.set_norm(norm)
    return {"case": case, "net": net, "x": x, "queries": queries}


def _run_choose(s):
    return {"predicted": s["net"].forward(s["x"]), "kappa": s["net"].invert_kappa(s["queries"])}


_PREPARE = {"run": _prepare_run, "batch": _prepare_batch, "train": _prepare_train,
            "choose": _prepare_choose}
_RUN = {"run": _run_run, "batch": _run_batch, "train": _run_train, "choose": _run_choose}


def prepare(case, seed):
    return _PREPARE[case["kind"]](case, seed)


def run(state):
    return _RUN[state["case"]["kind"]](state)


# --------------------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------------------

_FLOPS = 330           # of one site's update: moments, equilibria, forcing, sources, M^-1, EOS


def work(case):
    """A step reads and writes each population once; a diagnostic reads each once; a
    checkpoint reads each once and writes it once; a start reads three fields."""
    if case["kind"] == "run":
        s = {"fp64": 8, "fp32": 4, "bf16": 2}[case["prec"]]
        sites = case["nx"] * case["ny"]
        b = 18 * s * sites * case["steps"] + 18 * s * sites
        if case["read"] != "none":
            b += 9 * s * sites
        if case["resume"]:
            b += 18 * s * sites
        if case["state"] == "splash":
            b += (24 + 9 * s) * sites
        return {"bytes": b, "flops": _FLOPS * sites * case["steps"]}
    if case["kind"] == "batch":
        sizes = [r[0] ** 2 for r in _batch_rows(case)]
        n = 64 * case["ticks"]
        return {"bytes": sum(sizes) * (72 * n + 36 * case["ticks"]) + 72 * sizes[case["n"] // 2],
                "flops": _FLOPS * sum(sizes) * n}
    if case["kind"] == "train":
        mac = 64 * 3 + 64 * 64 + 3 * 64
        return {"bytes": case["steps"] * (24 * case["n"] + 26 * 4611),
                "flops": 6 * mac * case["n"] * case["steps"]}
    mac = 64 * 3 + 64 * 64 + 3 * 64
    return {"bytes": 40 * case["n"] + 2 * 4611, "flops": 2 * mac * case["n"] * 43}


# --------------------------------------------------------------------------------------
# the same outputs in 64 bits, plain torch
# --------------------------------------------------------------------------------------

_EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
_EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
_OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
_W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


def _moved(v, dx, dy, bc):
    """v(x - dx, y - dy) over the last two dimensions: periodic, or the nearest site's value
    beyond a wall (bc 1: in y) or an open side (bc 2: in x and y)."""
    for d, dim, wrap in ((dx, -1, bc != 2), (dy, -2, bc == 0)):
        if d == 0:
            continue
        if wrap:
            v = torch.roll(v, d, dim)
        else:
            i = torch.arange(v.shape[dim], device=v.device)
            v = v.index_select(dim, (i - d).clamp_(0, v.shape[dim] - 1))
    return v


def _psi(rho, p):
    if p["eos"] == "cs":
        eta = rho                      # b = 4
        pr = rho * p["T"] * (1 + eta + eta**2 - eta**3) / (1 - eta) ** 3 - rho**2
    else:
        v, m, l, r1, r2 = 0.49 / 3, -0.06 / 3, 1 / 3, 1.49, 94.65
        pr = torch.where(rho <= r1, rho * v,
                         torch.where(rho < r2, r1 * v + (rho - r1) * m,
                                     r1 * v + (r2 - r1) * m + (rho - r2) * l))
    return torch.sqrt(2 * (pr - rho / 3) / G)


def _equilibrium(rho, ux, uy):
    f = []
    u2 = ux * ux + uy * uy
    for a in range(9):
        eu = _EX[a] * ux + _EY[a] * uy
        f.append(_W[a] * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * u2))
    return f


def _forces(psi, bc):
    """Sums over the neighbours of psi: (S_x, S_y) of Eq. 7 and (xx, yy, xy) of Eq. 19."""
    nb = [_moved(psi, -_EX[a], -_EY[a], bc) for a in range(9)]
    diag = nb[5] + nb[6] + nb[7] + nb[8] - 4 * psi
    sx = (nb[1] - nb[3]) / 3 + (nb[5] - nb[6] - nb[7] + nb[8]) / 12
    sy = (nb[2] - nb[4]) / 3 + (nb[5] + nb[6] - nb[7] - nb[8]) / 12
    xx = (nb[1] + nb[3] - 2 * psi) / 3 + diag / 12
    yy = (nb[2] + nb[4] - 2 * psi) / 3 + diag / 12
    xy = (nb[5] - nb[6] + nb[7] - nb[8]) / 12
    return sx, sy, xx, yy, xy


def _step(f, p):
    """One time step of the update (Eqs. 1-8, 17-19) for populations f[a] of [..., ny, nx]."""
    bc = p["bc"]
    rho = f[0] + f[1] + f[2] + f[3] + f[4] + f[5] + f[6] + f[7] + f[8]
    psi = _psi(rho, p)
    sx, sy, xx, yy, xy = _forces(psi, bc)
    fx, fy = -G * psi * sx, -G * psi * sy
    q = p["kappa"] * (G / 2) * psi
    xx, yy, xy = q * xx, q * yy, q * xy
    ax, ay = f[1] + f[3], f[2] + f[4]
    s57, s68, d57, d68 = f[5] + f[7], f[6] + f[8], f[5] - f[7], f[6] - f[8]
    jx, jy = f[1] - f[3] + d57 - d68, f[2] - f[4] + d57 + d68
    vx, vy = (jx + fx / 2) / rho, (jy + fy / 2) / rho
    v2 = vx * vx + vy * vy
    s_e, s_q, s_v = 0.8, 1.1, p["s_v"]
    if "s_v_vapour" in p:
        s_v = torch.where(rho >= RHO_1, torch.full_like(rho, s_v),
                          torch.full_like(rho, p["s_v_vapour"]))
    s1 = 6 * (vx * fx + vy * fy)
    if p["sigma"]:
        s1 = s1 + 12 * p["sigma"] * (sx * sx + sy * sy) * G * G / (1 / s_e - 0.5)
    src = 1.5 * s_e * (xx + yy)

    def relax(s, m, meq, force):
        return m - s * (m - meq) + (1 - s / 2) * force

    e = relax(s_e, -4 * f[0] - ax - ay + 2 * (s57 + s68), rho * (3 * v2 - 2), s1) + src
    z = relax(s_e, 4 * f[0] - 2 * (ax + ay) + s57 + s68, rho * (1 - 3 * v2), -s1) - src
    qx = relax(s_q, -2 * (f[1] - f[3]) + d57 - d68, -rho * vx, -fx)
    qy = relax(s_q, -2 * (f[2] - f[4]) + d57 + d68, -rho * vy, -fy)
    pxx = relax(s_v, ax - ay, rho * (vx * vx - vy * vy), 2 * (vx * fx - vy * fy)) - s_v * (xx - yy)
    pxy = relax(s_v, s57 - s68, rho * vx * vy, vx * fy + vy * fx) - s_v * xy
    jx, jy = jx + fx, jy + fy
    out = []
    for a in range(9):
        ex, ey = _EX[a], _EY[a]
        n = ex * ex + ey * ey
        me, mz = (-4, -1, 2)[n], (4, -2, 1)[n]
        g = rho / 9 + (me / 36) * e + (mz / 36) * z
        if ex:
            g = g + (ex / 6) * jx + (ex * (-2, 1)[n - 1] / 12) * qx
        if ey:
            g = g + (ey / 6) * jy + (ey * (-2, 1)[n - 1] / 12) * qy
        if n == 1:
            g = g + ((ex * ex - ey * ey) / 4) * pxx
        if n == 2:
            g = g + (ex * ey / 4) * pxy
        out.append(g)
    new = [_moved(out[a], _EX[a], _EY[a], bc) for a in range(9)]
    if bc:                             # bounce-back from the wall below (and above: bc 1)
        for a in range(9):
            if _EY[a] == 1:
                new[a][..., 0, :] = out[_OPP[a]][..., 0, :]
            if _EY[a] == -1 and bc == 1:
                new[a][..., -1, :] = out[_OPP[a]][..., -1, :]
    return new


def _laplace(rho, psi, radius):
    """The eight numbers of a droplet measurement of one [ny][nx] lattice."""
    ny, nx = rho.shape
    y, x = _grid(nx, ny)
    r = torch.sqrt((x - 0.5 * (nx - 1)) ** 2 + (y - 0.5 * (ny - 1)) ** 2)
    inside, outside = r < 0.5 * radius, r > radius + 0.15 * min(nx, ny)
    pr = rho / 3 + 0.5 * G * psi * psi
    ri, ro, pi, po = (float(v[m].mean()) for v in (rho, pr) for m in (inside, outside))
    mass = float(rho.sum())
    big = math.sqrt((mass - ro * nx * ny) / (math.pi * (ri - ro)))
    return [(pi - po) * big, ri, ro, big, pi, po, mass, 0.0]


def _exact_run(case, seed):
    rho, ux, uy, radius = _fields(case, seed)
    mid = float(rho.max() + rho.min()) / 2
    p = {"bc": {"droplet": 0, "layer": 1, "splash": 2}[case["state"]], "kappa": case["kappa"],
         "sigma": 0.0, "eos": "cs", "s_v": _rates(case).s_v}
    if case["state"] == "splash":
        nu_v = 20.0 * 0.125 * 100.0 * _splash_scale(case) / 1000.0
        p.update(eos="piecewise", sigma=SIGMA_F, s_v_vapour=1.0 / (3.0 * nu_v + 0.5))
    else:
        p["T"] = lbm.cs_eos(case["t"]).T
    f = _equilibrium(rho, ux, uy)
    del ux, uy
    for _ in range(case["steps"]):
        f = _step(f, p)
    rho = sum(f)
    out = {}
    if case["read"] != "none":
        psi = _psi(rho, p)
    if case["read"] == "reduce":
        sx, sy = _forces(psi, p["bc"])[:2]
        px = f[1] - f[3] + f[5] - f[6] - f[7] + f[8] - G / 2 * psi * sx
        py = f[2] - f[4] + f[5] + f[6] - f[7] - f[8] - G / 2 * psi * sy
        out["sums"] = np.array([float(rho.sum()), float(px.sum()), float(py.sum()),
                                float((torch.hypot(px, py) / rho).max())])
    elif case["read"] == "droplet":
        out["droplet"] = np.array(_laplace(rho, psi, radius))
    elif case["read"] == "height":
        below = (rho < mid).to(torch.int8).argmax(0)
        r0 = rho.gather(0, (below - 1).clamp_min(0)[None])[0]
        r1 = rho.gather(0, below[None])[0]
        out["height"] = ((below - 1) + (r0 - mid) / (r0 - r1)).cpu().numpy()
    w = [v * _shift(case) for v in _W]
    out["populations"] = torch.stack([(f[a] - w[a]).cpu() for a in range(9)])
    return out


def _exact_batch(case, seed):
    rows, rho = _batch_density(case, seed)
    n, keep, pops = len(rows), case["n"] // 2, None
    out = np.zeros((case["ticks"], n, 8))
    for side in sorted({r[0] for r in rows}):
        mine = [i for i in range(n) if rows[i][0] == side]
        for k in range(0, len(mine), 64):
            ids = mine[k:k + 64]

            def col(vals):
                return torch.tensor(vals, dtype=torch.float64, device="cuda")[:, None, None]

            p = {"bc": 0, "sigma": SIGMA_F, "eos": "cs",
                 "T": col([lbm.cs_eos(rows[i][1]).T for i in ids]),
                 "kappa": col([rows[i][2] for i in ids]),
                 "s_v": col([1.0 / rows[i][3] for i in ids])}
            r = torch.stack([rho[i] for i in ids])
            f = _equilibrium(r, torch.zeros_like(r), torch.zeros_like(r))
            for tick in range(case["ticks"]):
                for _ in range(64):
                    f = _step(f, p)
                r = sum(f)
                psi = _psi(r, p)
                for j, i in enumerate(ids):
                    out[tick, i] = _laplace(r[j], psi[j], rows[i][4])
            if keep in ids:
                pops = torch.stack([v[ids.index(keep)] for v in f]).cpu().numpy()
    return {"readings": out, "populations": pops}


def _net(theta, norm, x):
    """(predictions, activations) of the 3-64-64-3 network in 64 bits; the weights are the
    BF16 values nearest to theta's."""
    t = torch.as_tensor(np.asarray(theta), device="cuda").to(torch.float32)
    t = t.to(torch.bfloat16).to(torch.float64)
    w1, b1, w2, b2, w3, b3 = torch.split(t, [192, 64, 4096, 64, 192, 3])
    im, isc, om, osc = (torch.as_tensor(np.asarray(v), device="cuda").double() for v in norm)
    x = torch.as_tensor(np.asarray(x), device="cuda").double()
    xn = (torch.stack([torch.log1p(-x[:, 0]), torch.log1p(-x[:, 1]), x[:, 2]], 1) - im) / isc
    z1 = xn @ w1.view(64, 3).T + b1
    a1 = z1 * _phi(z1)
    z2 = a1 @ w2.view(64, 64).T + b2
    a2 = z2 * _phi(z2)
    o = a2 @ w3.view(3, 64).T + b3
    y = o * osc + om
    return torch.stack([y[:, 0].exp(), y[:, 1], y[:, 2].exp()], 1), (xn, z1, a1, z2, a2, o, w2, w3)


def _phi(z):
    return 0.5 * (1 + torch.erf(z / math.sqrt(2)))


def _slope(z):
    return _phi(z) + z * torch.exp(-z * z / 2) / math.sqrt(2 * math.pi)


def _exact_train(case, seed):
    x, y = _samples(case["n"], seed)
    xd, yd = x.astype(np.float64), y.astype(np.float64)
    feat = np.stack([np.log1p(-xd[:, 0]), np.log1p(-xd[:, 1]), xd[:, 2]], 1)
    tgt = np.stack([np.log(yd[:, 0]), yd[:, 1], np.log(yd[:, 2])], 1)
    norm = [feat.mean(0), feat.std(0), tgt.mean(0), tgt.std(0)]
    tn = torch.as_tensor((tgt - norm[2]) / norm[3], device="cuda")
    theta = torch.as_tensor(inputs.mlp_init(seed).astype(np.float64), device="cuda")
    m, v = torch.zeros_like(theta), torch.zeros_like(theta)
    loss = 0.0
    for k in range(1, case["steps"] + 1):
        _, (xn, z1, a1, z2, a2, o, w2, w3) = _net(theta.cpu().numpy(), norm, x)
        r = o - tn
        loss = float((r * r).mean())
        do = 2 * r / r.numel()
        d2 = (do @ w3.view(3, 64)) * _slope(z2)
        d1 = (d2 @ w2.view(64, 64)) * _slope(z1)
        g = torch.cat([(d1.T @ xn).ravel(), d1.sum(0), (d2.T @ a1).ravel(), d2.sum(0),
                       (do.T @ a2).ravel(), do.sum(0)])
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        theta = theta - _LR * (m / (1 - 0.9**k)) / ((v / (1 - 0.999**k)).sqrt() + 1e-8)
    return {"loss": np.array([loss]), "params": theta.cpu().numpy()}


def _exact_choose(case, seed):
    theta, norm, x, queries = _choose_inputs(case, seed)
    q = queries.astype(np.float64)
    lo, hi = np.zeros(len(q)), np.full(len(q), 0.95)
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        high = _net(theta, norm, np.stack([q[:, 0], mid, q[:, 1]], 1))[0][:, 0]
        up = high.cpu().numpy() > q[:, 2]
        lo, hi = np.where(up, mid, lo), np.where(up, hi, mid)
    return {"predicted": _net(theta, norm, x)[0].cpu().numpy(),
            "kappa": 0.5 * (lo + hi)}


_EXACT = {"run": _exact_run, "batch": _exact_batch, "train": _exact_train,
          "choose": _exact_choose}


def exact(case, seed):
    return _EXACT[case["kind"]](case, seed)
