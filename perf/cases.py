"""The work a user has this library do, as cases that can be timed and compared.

Three kinds of case, each through the package's public entry points:

  channel  one channel (or drop box) stepped by `Lbm`: a number of time steps, then the
           macroscopic fields, as device tensors or (the drop study's sampling loop) as host
           arrays;
  sweep    many channels stepped together by `LbmBatch` in chunks of 100 steps with their
           residual checks, then every channel's fields in float32, as the warm-start
           surrogate's training set holds them;
  cnn      the warm-start surrogate `Cnn`: a prediction, a gradient, or one training step.

Sizes are those of the repository's own workloads, tests and benchmark, and odd or ragged
ones of the same ranges.  Channels start from a slightly displaced tanh interface, a smooth
velocity (FP64: at rest) and a heated temperature profile: the state of a channel under way (from
the default start the velocity would stay at round-off until the heat reaches the interface).

`exact` restates the method in plain float64 torch: streaming with the wall rules, central
moments, relaxation (arXiv 2210.07501, Sec. 4, Sec. 5.1, App. B), and the surrogate's network.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2210_07501_gb300 as lbm

CHECK = 100            # steps per residual check of a sweep (the library's default)
FIELDS = ("phi", "u", "v", "T", "dp")
CH = (12, 32, 32, 32, 32, 32, 4)   # channels of the surrogate's layers
LR = 1e-3

PARAMS = dict(sigma0=1e-3, sigma1=0.0, sigma2=-1e-4, T_ref=1.0, T_hot=1.0, T_cold=1.0, dT=1.0, tau_flow=0.8,
              visc_ratio=1.0, tau_T=0.8, cond_ratio=1.0, tau_phi=0.8, rho_bottom=1.0, rho_top=1.0, Fx_ext=0.0,
              Fy_ext=0.0)


# ---- the cases ---------------------------------------------------------------------------
def _channel(nx, ny, b, precision, steps, W=5.0, heat_periods=1, q_phi=5, q_T=5, read="device", tune=False,
             **params):
    return {"kind": "channel", "nx": nx, "ny": ny, "b": float(b), "W": float(W), "heat_periods": heat_periods,
            "q_phi": q_phi, "q_T": q_T, "precision": precision, "steps": steps, "read": read, "tune": tune, **params}


def listed():
    return [
        # the smallest workload: the plain 128 x 32 channel, where launches and latency count
        dict(_channel(128, 32, 16, "fp32", 50, W=4.0), name="channel 128x32 fp32"),
        # the paper's validation channel of the parametric studies, all lattices D2Q9, FP64
        dict(_channel(200, 100, 50, "fp64", 30, q_phi=9, q_T=9, sigma0=1e-2, sigma2=1e-3, tau_phi=0.56,
                      tau_flow=1.17, tau_T=2.73), name="paper channel 200x100 fp64"),
        # the drop migration study: steps between two samples, fields read into host arrays
        dict(_channel(160, 320, 160, "fp64", 30, q_phi=9, q_T=9, read="host", sigma0=2.5e-3, sigma1=-1e-4,
                      sigma2=0.0, T_ref=16.0, T_hot=0.0, T_cold=32.0, dT=0.0, tau_flow=1.1, tau_T=1.1,
                      tau_phi=0.56), name="drop 160x320 fp64"),
        # the run to a steady state, tuned once: 100 steps, the residual check and its diagnosis
        dict(_channel(1024, 256, 128, "fp32", 100, read="diag", tune=True, sigma2=-2e-4, visc_ratio=2.0, cond_ratio=2.0),
             name="steady channel 1024x256 fp32"),
        # the same channel in FP64 (the reference run of the steady state)
        dict(_channel(1024, 256, 128, "fp64", 20, sigma2=-2e-4, visc_ratio=2.0, cond_ratio=2.0),
             name="steady channel 1024x256 fp64"),
        # a ragged channel with unequal lattices and every option on
        dict(_channel(523, 187, 80.3, "fp32", 40, W=4.0, heat_periods=2, q_phi=9, q_T=5, sigma0=2e-3, sigma1=-3e-5,
                      sigma2=5e-5, T_hot=1.2, T_cold=0.9, dT=0.6, tau_flow=0.9, visc_ratio=1.7, tau_T=1.1,
                      cond_ratio=0.6, tau_phi=0.75, rho_top=1.3, Fx_ext=2e-8),
             name="ragged channel 523x187 fp32"),
        # the bandwidth workload, tuned as the benchmark does
        dict(_channel(8192, 2048, 1365, "fp32", 20, heat_periods=4, tune=True), name="channel 8192x2048 fp32"),
        # half the memory per node: FP16 storage, FP32 arithmetic
        dict(_channel(8192, 1024, 683, "fp16", 10, heat_periods=4), name="channel 8192x1024 fp16"),
        # the parameter sweep: channels of uneven size to a common number of steps
        {"name": "sweep of 12 uneven fp32", "kind": "sweep", "cases": 12, "uneven": True, "nx": 1024, "ny": 256,
         "precision": "fp32", "steps": 300, "pick": 0},
        # training channels of the surrogate: one grid, many parameter sets
        {"name": "sweep of 32 256x64 fp32", "kind": "sweep", "cases": 32, "uneven": False, "nx": 256, "ny": 64,
         "precision": "fp32", "steps": 300, "pick": 1},
        # one training step of the surrogate at its training batch
        {"name": "cnn train 16x256x64", "kind": "cnn", "do": "train", "H": 64, "W": 256, "B": 16, "bf16": True},
        # its prediction for a batch of small channels
        {"name": "cnn predict 16x64x32", "kind": "cnn", "do": "predict", "H": 32, "W": 64, "B": 16, "bf16": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.random()
    if what < 0.6:
        precision = rng.choice(["fp32", "fp32", "fp32", "fp64", "fp64", "fp16"])
        nx = _log_int(rng, 48, 8192)
        ny = _log_int(rng, 24, 2048)
        if precision == "fp64":                       # FP64 work costs ~25 times as much per node
            ny = max(24, min(ny, (1 << 19) // nx))
        nodes = nx * ny
        steps = 50 if nodes <= 1 << 18 else (20 if nodes <= 1 << 20 else 10)
        if precision == "fp64":
            steps = 30 if nodes <= 1 << 16 else 20
        if precision == "fp16":
            steps = 10
        q = rng.choice([(5, 5), (5, 5), (9, 9), (9, 5), (5, 9)])
        return _channel(nx, ny, round(ny * rng.uniform(0.3, 0.7), 1), precision, steps, W=rng.choice([4.0, 5.0]),
                        heat_periods=rng.choice([1, 2, 4]), q_phi=q[0], q_T=q[1], tune=rng.random() < 0.5,
                        sigma1=rng.uniform(-2e-5, 2e-5), sigma2=rng.uniform(-4e-4, 0.0),
                        visc_ratio=rng.uniform(0.5, 4.0), cond_ratio=rng.uniform(0.5, 4.0),
                        rho_top=rng.choice([1.0, 1.0, 1.3]))
    if what < 0.8:
        uneven = rng.random() < 0.5
        nx, ny = (1024, 256) if uneven else (_log_int(rng, 64, 512), _log_int(rng, 32, 128))
        return {"kind": "sweep", "cases": rng.randint(3, 12) if uneven else rng.randint(6, 32), "uneven": uneven, "nx": nx,
                "ny": ny, "precision": "fp32", "steps": 200, "pick": rng.randrange(1, 1 << 20)}
    do = rng.choice(["train", "predict", "gradient"])
    H, W = _log_int(rng, 20, 96), _log_int(rng, 32, 256)
    return {"kind": "cnn", "do": do, "H": H, "W": W, "B": rng.randint(1, 16 if H * W <= 16384 else 8),
            "bf16": rng.random() < 0.6}


# ---- inputs ------------------------------------------------------------------------------
def _split(case):
    domain = {k: case[k] for k in ("nx", "ny", "b", "W", "heat_periods", "q_phi", "q_T")}
    return domain, {**PARAMS, **{k: v for k, v in case.items() if k in PARAMS}}


def _sweep_cases(case):
    """The sweep's channels: sigma1, sigma2, a/b and both ratios uniform; sizes uneven or one grid."""
    rng = np.random.Generator(np.random.PCG64(case["pick"]))
    out = []
    for _ in range(case["cases"]):
        nx, ny = case["nx"], case["ny"]
        if case["uneven"]:
            nx, ny = int(rng.choice([nx // 4, nx // 2, nx])), int(rng.choice([ny // 4, ny // 2, ny]))
        ab = rng.uniform(0.25, 4.0)
        b = min(max(round(ny / (1.0 + ab)), 3), ny - 3)
        out.append(_channel(nx, ny, b, case["precision"], case["steps"], sigma1=float(rng.uniform(-2e-5, 2e-5)),
                            sigma2=float(rng.uniform(-4e-4, 0.0)), cond_ratio=float(rng.uniform(0.5, 4.0)),
                            visc_ratio=float(rng.uniform(0.5, 4.0))))
    return out


def _start(case, seed):
    """Fields [ny][nx]: the interface displaced by a few hundredths of a node, the wall heating faded
    towards the top and a smooth temperature on it.  FP64 channels start at rest and uniform p, as
    the studies that use FP64 do; the others are under way, with convection cells and a smooth p (a
    small one over longer passes: sound moves phi off 1 in the bulk, where the unit normal is then
    undefined along every extremum and rounding grows)."""
    domain, p = _split(case)
    nx, ny = domain["nx"], domain["ny"]
    rng = np.random.Generator(np.random.PCG64(seed))
    x = np.arange(nx) / nx
    y = (np.arange(ny) + 0.5) / ny

    def smooth(amp):
        f = np.zeros((ny, nx))
        for _ in range(3):
            kx, ky, ph = int(rng.integers(1, 4)), int(rng.integers(1, 4)), rng.uniform(0, 2 * np.pi)
            f += np.outer((0.5 + rng.random()) * amp * np.sin(np.pi * ky * y), np.cos(2 * np.pi * kx * x + ph))
        return f

    def cells(amp):
        """Divergence-free convection cells that vanish at the walls: psi ~ sin^2(pi ky y) cos(kx x)."""
        u, v = np.zeros((ny, nx)), np.zeros((ny, nx))
        for _ in range(3):
            kx, ky, ph = int(rng.integers(1, 4)), int(rng.integers(1, 3)), rng.uniform(0, 2 * np.pi)
            a, r = (0.5 + rng.random()) * amp, 2.0 * kx * ny / (ky * nx)     # r: v against u
            a /= max(1.0, r)
            u += np.outer(a * np.sin(2 * np.pi * ky * y), np.cos(2 * np.pi * kx * x + ph))
            v += np.outer(a * r * np.sin(np.pi * ky * y) ** 2, np.sin(2 * np.pi * kx * x + ph))
        return u, v

    wave = np.zeros(nx)
    for k in (1, 2, 3):
        wave += rng.uniform(0.01, 0.03) * np.sin(2 * np.pi * k * x + rng.uniform(0, 2 * np.pi))
    if case["read"] == "host":      # the drop study: a drop of radius nx / 8, a little off a circle
        dx, dy = (np.arange(nx) - nx / 2.0)[None, :], (np.arange(ny) + 0.5 - ny / 2.0)[:, None]
        r = np.sqrt(dx ** 2 + dy ** 2)
        R = nx / 8.0 + rng.uniform(-0.3, 0.3) + 0.2 * np.cos(2 * np.arctan2(dy, dx) + rng.uniform(0, 2 * np.pi))
        phi = 0.5 + 0.5 * np.tanh(2.0 * (R - r) / domain["W"])
        T = (p["T_hot"] + (p["T_cold"] - p["T_hot"]) * y)[:, None] + smooth(0.05)
        return dict(phi=phi, u=None, v=None, T=T, dp=None)
    phi = np.tanh(2.0 * ((np.arange(ny) + 0.5 - domain["b"])[:, None] - wave[None, :]) / domain["W"])
    phi = 0.5 + 0.5 * phi
    heat = p["T_hot"] - p["T_cold"] + p["dT"] * np.cos(2 * np.pi * domain["heat_periods"] * x)
    T = p["T_cold"] + np.outer(1.0 - y, heat) + smooth(0.05 * abs(p["dT"]))
    if case["precision"] == "fp64":
        return dict(phi=phi, u=None, v=None, T=T, dp=None)
    u, v = cells(1e-4)
    return dict(phi=phi, u=u, v=v, T=T, dp=smooth(2e-5 if case["steps"] <= 50 else 1e-6))


def _cnn_inputs(case, seed):
    """Inputs like the surrogate's (profiles over the grid, constant parameter channels), smooth targets
    and He-style weights; float32 arrays."""
    rng = np.random.Generator(np.random.PCG64(seed))
    B, H, W = case["B"], case["H"], case["W"]
    x = np.broadcast_to(np.arange(W) / W, (H, W))
    y = np.broadcast_to(((np.arange(H) + 0.5) / H)[:, None], (H, W))
    X, Y = np.empty((B, CH[0], H, W), np.float32), np.empty((B, CH[-1], H, W), np.float32)
    c, s = np.cos(2 * np.pi * x), np.sin(2 * np.pi * x)
    for n in range(B):
        b = rng.uniform(0.2, 0.8)
        for k, v in enumerate((c, s, y, (y < b).astype(float), y - b, 0.5 + 0.5 * np.tanh(0.4 * H * (y - b)),
                               c * (1.0 - y))):
            X[n, k] = v
        for k in range(7, CH[0]):
            X[n, k] = rng.uniform(-1.0, 1.0)
        for k in range(CH[-1]):
            Y[n, k] = rng.normal() * c * np.sin(np.pi * y) + rng.normal() * s * np.sin(2 * np.pi * y) \
                + 0.1 * rng.normal()
    flat = []
    for l in range(len(CH) - 1):
        flat.append(rng.uniform(-1, 1, CH[l + 1] * CH[l] * 9) * math.sqrt(6.0 / (CH[l] * 9)))
        flat.append(rng.uniform(-0.1, 0.1, CH[l + 1]))
    return X, Y, np.concatenate(flat).astype(np.float32)


_streams = []


def _stream():
    """One stream for the program's tensors and the library's kernels, as the warm-start pipeline has."""
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


def prepare(case, seed):
    stream = _stream()
    with torch.cuda.stream(stream):
        if case["kind"] == "channel":
            domain, params = _split(case)
            g = lbm.Lbm(domain, params, precision=case["precision"], stream=stream)
            g.lbm_init_fields(**_start(case, seed))
            if case["tune"]:
                g.lbm_autotune(2)
            dt = torch.float64 if case["precision"] == "fp64" else torch.float32
            out = {} if case["read"] == "host" else {k: torch.empty((case["ny"], case["nx"]), dtype=dt, device="cuda")
                                                     for k in FIELDS}
            return {"case": case, "g": g, "out": out}
        if case["kind"] == "sweep":
            cases = _sweep_cases(case)
            b = lbm.LbmBatch([dict(zip(("domain", "params"), _split(c))) for c in cases],
                             precision=case["precision"], stream=stream)
            b.lbm_batch_set_check_interval(CHECK)
            for c, w in enumerate(cases):
                b.lbm_batch_init_fields(c, **_start(w, seed * 1000 + c))
            b.lbm_batch_autotune(3)      # as the sweep and the warm-start pipeline do
            return {"case": case, "b": b}
        X, Y, flat = _cnn_inputs(case, seed)
        net = lbm.Cnn(case["H"], case["W"], batch_max=case["B"], bf16=case["bf16"], stream=stream)
        net.set_params(flat)
        st = {"case": case, "net": net, "x": torch.tensor(X, device="cuda")}
        if case["do"] == "predict":
            st["y"] = torch.empty(Y.shape, dtype=torch.float32, device="cuda")
        else:
            st["t"] = torch.tensor(Y, device="cuda")
        stream.synchronize()
        return st


# ---- one pass ----------------------------------------------------------------------------
def run(state):
    case = state["case"]
    if case["kind"] == "channel":
        g, out = state["g"], state["out"]
        g.lbm_step(case["steps"])
        if case["read"] == "host":
            return g.lbm_fields()
        res = {}
        if case["read"] == "diag":      # as lbm_run_to_steady reads it after each check interval
            d = g.lbm_diag()
            res = {"mass": d["mass"], "residual": d["residual"]}
        g.lbm_fields_device(**out, dtype=lbm.LBM_DTYPE_F64 if case["precision"] == "fp64" else lbm.LBM_DTYPE_F32)
        return {**out, **res}
    if case["kind"] == "sweep":
        b = state["b"]
        b.lbm_batch_step(case["steps"])
        got = [b.lbm_batch_fields(c) for c in range(b.n)]
        residual = np.array([b.lbm_batch_diag(c)["residual"] for c in range(b.n)], dtype=np.float32)
        if case["uneven"]:
            return {"residual": residual, "fields": [{k: f[k].astype(np.float32) for k in FIELDS} for f in got]}
        return {"residual": residual, "fields": {k: np.stack([f[k].astype(np.float32) for f in got]) for k in FIELDS}}
    net = state["net"]
    if case["do"] == "predict":
        net.forward(state["x"], state["y"])
        return state["y"]
    if case["do"] == "gradient":
        grad, loss = net.gradients(state["x"], state["t"])
        return {"grad": grad, "loss": loss}
    loss = net.train_step(state["x"], state["t"], LR)
    return {"loss": loss, "params": net.get_params()}


# ---- what a pass cannot do without -------------------------------------------------------
def work(case):
    """A step reads and writes every population and the stored pressure once; arithmetic as
    the collisions need it (about 500 operations a node, 100 more per D2Q9 scalar lattice)."""
    if case["kind"] in ("channel", "sweep"):
        bytes_, flops = 0.0, 0.0
        for c in ([case] if case["kind"] == "channel" else _sweep_cases(case)):
            s, r = {"fp64": (8, 8), "fp32": (4, 4), "fp16": (2, 4)}[c["precision"]]
            n = c["nx"] * c["ny"]
            bytes_ += n * (c["steps"] * (2 * (c["q_phi"] + 9 + c["q_T"]) * s + 2 * r) + len(FIELDS) * r)
            flops += n * c["steps"] * (500.0 + 25.0 * (c["q_phi"] + c["q_T"] - 10))
        return {"bytes": bytes_, "flops": flops}
    px = case["B"] * case["H"] * case["W"]
    macs = sum(CH[l] * CH[l + 1] * 9 for l in range(len(CH) - 1))
    n_params = macs + sum(CH[1:])
    if case["do"] == "predict":
        return {"bytes": 4.0 * (px * (CH[0] + CH[-1]) + n_params), "flops": 2.0 * px * macs}
    return {"bytes": 4.0 * (px * (CH[0] + CH[-1]) + (2 if case["do"] == "gradient" else 7) * n_params),
            "flops": 2.0 * px * (3 * macs - CH[0] * CH[1] * 9)}


# ---- the same in 64 bits -----------------------------------------------------------------
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
ORDER = ((0, 0), (1, 0), (0, 1), (2, 0), (0, 2), (1, 1), (2, 1), (1, 2), (2, 2))
C2 = 1.0 / 3.0


def _weights(Q):
    return [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4 if Q == 9 else [1 / 3] + [1 / 6] * 4


def _find(Q, ex, ey):
    return next(a for a in range(Q) if EX[a] == ex and EY[a] == ey)


def _populations(k, ux, uy, Q):
    """Central moments {(m, n): value} -> populations: raw moments by the binomial expansion about u,
    then the inverse of the moment matrix, written per direction (App. B)."""
    px, py = (1.0, ux, ux * ux), (1.0, uy, uy * uy)
    r = {}
    for m, n in ORDER[:Q]:
        v = 0.0
        for a in range(m + 1):
            for b in range(n + 1):
                if (a, b) in k:
                    v = v + math.comb(m, a) * math.comb(n, b) * px[m - a] * py[n - b] * k[a, b]
        r[m, n] = v
    if Q == 5:
        return torch.stack([r[0, 0] - r[2, 0] - r[0, 2], (r[1, 0] + r[2, 0]) / 2, (r[0, 1] + r[0, 2]) / 2,
                            (r[2, 0] - r[1, 0]) / 2, (r[0, 2] - r[0, 1]) / 2])
    out = []
    for a in range(9):
        ix = [(0, 1.0), (2, -1.0)] if EX[a] == 0 else [(1, EX[a] / 2), (2, 0.5)]
        iy = [(0, 1.0), (2, -1.0)] if EY[a] == 0 else [(1, EY[a] / 2), (2, 0.5)]
        out.append(sum(cx * cy * r[m, n] for m, cx in ix for n, cy in iy))
    return torch.stack(out)


def _pull(P, rule, wall=None):
    """Streamed populations; at a wall: specular reflection ('free'), bounce-back ('no slip'), or
    anti-bounce-back to the wall temperature where the link crosses it ('heat')."""
    Q = P.shape[0]
    out = torch.empty_like(P)
    for a in range(Q):
        ex, ey = EX[a], EY[a]
        src = torch.roll(P[a], ex, 1)
        if ey == 0:
            out[a] = src
            continue
        row, inside, from_ = (0, slice(1, None), slice(None, -1)) if ey > 0 else (-1, slice(None, -1), slice(1, None))
        out[a][inside] = src[from_]
        if rule == "free":
            out[a][row] = torch.roll(P[_find(Q, ex, -ey)][row], ex, 0)
        else:
            back = P[_find(Q, -ex, -ey)][row]
            out[a][row] = back if rule == "no slip" else 2 * _weights(Q)[a] * wall(ex, ey) - back
    return out


def _pad(f, rows, top=None, bottom=None):
    """Ghost rows: mirrored, or 2 wall - adjacent where wall values are given; periodic columns."""
    lo = torch.flip(f[:rows], (0,)) if bottom is None else (2 * bottom - f[0])[None]
    hi = torch.flip(f[-rows:], (0,)) if top is None else (2 * top - f[-1])[None]
    f = torch.cat([lo, f, hi])
    return torch.cat([f[:, -1:], f, f[:, :1]], 1)


def _gradient(f):
    """Isotropic differences with the D2Q9 weights, of a field padded by one on every side."""
    c, r, l = f[:, 1:-1], f[:, 2:], f[:, :-2]
    gx = (r - l)[1:-1] / 3 + ((r - l)[2:] + (r - l)[:-2]) / 12
    gy = (c[2:] - c[:-2]) / 3 + ((r + l)[2:] - (r + l)[:-2]) / 12
    return gx, gy


def _normals(phi):
    """Unit normals on the rows -1 .. ny (phi mirrored beyond the walls)."""
    gx, gy = _gradient(_pad(phi, 2))
    g2 = gx * gx + gy * gy
    some = g2 > 1e-24
    inv = torch.where(some, 1.0 / torch.sqrt(torch.where(some, g2, torch.ones_like(g2))), torch.zeros_like(g2))
    return gx * inv, gy * inv


def _flow_moments(dp, rho, ux, uy):
    """Equilibrium central moments of the pressure lattice minus those of the weights times p0."""
    ax, ay, rc2 = C2 + ux * ux, C2 + uy * uy, rho * C2
    d = rc2 - dp
    return {(0, 0): dp, (1, 0): ux * d, (0, 1): uy * d, (2, 0): dp * ax - rc2 * ux * ux,
            (0, 2): dp * ay - rc2 * uy * uy, (1, 1): -ux * uy * d, (2, 1): ax * uy * d, (1, 2): ay * ux * d,
            (2, 2): dp * ax * ay - rc2 * (C2 * (ux * ux + uy * uy) + ux * ux * uy * uy)}


def _heat_moments(dT, first, Tr, ux, uy):
    """Energy lattice minus T_ref times the weights: given first moments, the rest at equilibrium."""
    ux2, uy2 = ux * ux, uy * uy
    return {(0, 0): dT, (1, 0): first[0], (0, 1): first[1], (2, 0): C2 * dT - Tr * ux2, (0, 2): C2 * dT - Tr * uy2,
            (1, 1): -Tr * ux * uy, (2, 1): Tr * (C2 + ux2) * uy, (1, 2): Tr * (C2 + uy2) * ux,
            (2, 2): C2 * C2 * dT - Tr * (C2 * (ux2 + uy2) + ux2 * uy2)}


def _phase_moments(phi, first):
    return {(0, 0): phi, (1, 0): first[0], (0, 1): first[1], (2, 0): C2 * phi, (0, 2): C2 * phi,
            (2, 2): C2 * C2 * phi}


def _exact_channel(case, seed, device):
    """The channel's fields after case['steps'] steps."""
    domain, p = _split(case)
    nx, ny, Qf, Qh, W = domain["nx"], domain["ny"], domain["q_phi"], domain["q_T"], domain["W"]
    f0 = {k: torch.zeros((ny, nx), dtype=torch.float64, device=device) if v is None else
          torch.tensor(np.ascontiguousarray(v), dtype=torch.float64, device=device)
          for k, v in _start(case, seed).items()}
    Tr, om_phi = p["T_ref"], 1.0 / p["tau_phi"]
    M = (p["tau_phi"] - 0.5) / 3
    mu_b, k_b = p["rho_bottom"] * (p["tau_flow"] - 0.5) / 3, p["rho_bottom"] * (p["tau_T"] - 0.5) / 3
    drho = p["rho_top"] - p["rho_bottom"]
    xs = torch.arange(nx, dtype=torch.float64, device=device)

    def hot(shift):
        return p["T_hot"] + p["dT"] * torch.cos(2 * math.pi * domain["heat_periods"] * (xs + shift) / nx) - Tr

    walls = {ex: hot(-0.5 * ex) for ex in (-1, 0, 1)}
    cold = torch.full((nx,), p["T_cold"] - Tr, dtype=torch.float64, device=device)

    def wall(ex, ey):
        return walls[ex] if ey > 0 else cold

    phi, ux, uy, dT, dp = f0["phi"], f0["u"], f0["v"], f0["T"] - Tr, f0["dp"]
    n_x, n_y = _normals(phi)
    theta = 4 * phi * (1 - phi) / W
    f = _populations(_phase_moments(phi, (M * theta * n_x[1:-1], M * theta * n_y[1:-1])), ux, uy, Qf)
    g = _populations(_flow_moments(dp, p["rho_bottom"] + phi * drho, ux, uy), ux, uy, 9)
    h = _populations(_heat_moments(dT, (Tr * ux, Tr * uy), Tr, ux, uy), ux, uy, Qh)

    def step(f, g, h, dp_old):
        f, g, h = _pull(f, "free"), _pull(g, "no slip"), _pull(h, "heat", wall)
        phi, dT = f.sum(0), h.sum(0)
        n_x, n_y = _normals(phi)
        gx, gy = _gradient(_pad(phi, 1))
        dsx, dsy = _gradient(_sigma(_pad(dT, 1, cold, walls[0]), p))
        dpx, dpy = _gradient(_pad(dp_old, 1))
        wrap = lambda a: torch.cat([a[:, -1:], a, a[:, :1]], 1)  # noqa: E731
        div = _gradient(wrap(n_x))[0] + _gradient(wrap(n_y))[1]
        n_x, n_y = n_x[1:-1], n_y[1:-1]
        g2, csf = gx * gx + gy * gy, 1.5 * W
        sigma = p["sigma0"] + _sigma(dT, p)
        Fx = csf * g2 * (-sigma * div * n_x + (1 - n_x * n_x) * dsx - n_x * n_y * dsy) + p["Fx_ext"]
        Fy = csf * g2 * (-sigma * div * n_y + (1 - n_y * n_y) * dsy - n_x * n_y * dsx) + p["Fy_ext"]
        Px, Py = -dpx + C2 * drho * gx, -dpy + C2 * drho * gy
        rho = p["rho_bottom"] + phi * drho
        first = lambda P: (sum(EX[a] * P[a] for a in range(P.shape[0]) if EX[a]),   # noqa: E731
                           sum(EY[a] * P[a] for a in range(P.shape[0]) if EY[a]))
        sx, sy = first(g)
        ux, uy = (sx + C2 * Fx / 2) / (rho * C2), (sy + C2 * Fy / 2) / (rho * C2)
        s0 = g.sum(0)
        G = Px * ux + Py * uy
        dp = s0 + G / 2
        om_nu = 1 / (3 * (mu_b + phi * (p["visc_ratio"] - 1) * mu_b) / rho + 0.5)
        om_T = 1 / (3 * (k_b + phi * (p["cond_ratio"] - 1) * k_b) / rho + 0.5)
        theta = 4 * phi * (1 - phi) / W
        m = first(f)
        f = _populations(_phase_moments(phi, tuple((1 - om_phi) * (m[i] - (ux, uy)[i] * phi)
                                                   + om_phi * M * theta * (n_x, n_y)[i] for i in (0, 1))), ux, uy, Qf)
        m = first(h)
        q = tuple(m[i] - (ux, uy)[i] * dT for i in (0, 1))
        h = _populations(_heat_moments(dT, tuple(q[i] + om_T * (Tr * (ux, uy)[i] - q[i]) for i in (0, 1)), Tr, ux, uy),
                         ux, uy, Qh)
        # flow: trace-free second moments relax at om_nu, all others take equilibrium + source / 2
        e20 = sum(g[a] for a in range(9) if EX[a]) - 2 * ux * sx + ux * ux * s0
        e02 = sum(g[a] for a in range(9) if EY[a]) - 2 * uy * sy + uy * uy * s0
        e11 = sum(EX[a] * EY[a] * g[a] for a in range(5, 9)) - uy * sx - ux * sy + ux * uy * s0
        k = _flow_moments(dp, rho, ux, uy)
        ax, ay = C2 + ux * ux, C2 + uy * uy
        s20, s02 = 2 * C2 * Px * ux + ax * G, 2 * C2 * Py * uy + ay * G
        s11 = C2 * (Px * uy + Py * ux) + ux * uy * G
        trace = k[2, 0] + k[0, 2] + (s20 + s02) / 2
        diff = e20 - e02 + om_nu * (k[2, 0] - k[0, 2] - e20 + e02) + (1 - om_nu / 2) * (s20 - s02)
        k[1, 1] = e11 + om_nu * (k[1, 1] - e11) + (1 - om_nu / 2) * s11
        k[2, 0], k[0, 2] = (trace + diff) / 2, (trace - diff) / 2
        k[0, 0] = dp + G / 2
        k[1, 0] = k[1, 0] + (C2 * Fx - ux * G) / 2
        k[0, 1] = k[0, 1] + (C2 * Fy - uy * G) / 2
        g = _populations(k, ux, uy, 9)
        return f, g, h, dp, (phi, ux, uy, Tr + dT, dp)

    state = [f, g, h, dp]
    if device.type != "cuda" or nx * ny > 1 << 20:
        for _ in range(case["steps"]):
            *state, out = step(*state)
        return dict(zip(FIELDS, out))
    # small channels: one step as a graph of its several hundred tensor operations
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        step(*state)
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        *new, out = step(*state)
        for a, b in zip(state, new):
            a.copy_(b)
    for _ in range(case["steps"]):
        graph.replay()
    torch.cuda.synchronize()
    return {k: v.clone() for k, v in zip(FIELDS, out)}


def _sigma(dT, p):
    return dT * (p["sigma1"] + p["sigma2"] * dT)


def _exact_cnn(case, seed, device):
    X, Y, flat = (torch.tensor(a, dtype=torch.float64, device=device) for a in _cnn_inputs(case, seed))
    flat.requires_grad_(case["do"] != "predict")
    a, at = X, 0
    for l in range(len(CH) - 1):
        n = CH[l + 1] * CH[l] * 9
        w, b = flat[at:at + n].view(CH[l + 1], CH[l], 3, 3), flat[at + n:at + n + CH[l + 1]]
        at += n + CH[l + 1]
        a = torch.cat([a[..., -1:], a, a[..., :1]], -1)
        z = torch.nn.functional.conv2d(a, w, b, padding=(1, 0))
        a = z * torch.sigmoid(z) if l < len(CH) - 2 else z
    if case["do"] == "predict":
        return a
    loss = ((a - Y) ** 2).mean()
    (grad,) = torch.autograd.grad(loss, flat)
    flat = flat.detach()
    if case["do"] == "gradient":
        return {"grad": grad, "loss": float(loss.detach())}
    # the first Adam step: the moments' bias corrections cancel (g / (|g| + eps))
    return {"loss": float(loss.detach()), "params": flat - LR * grad / (grad.abs() + 1e-8)}


def exact(case, seed):
    device = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if case["kind"] == "cnn":
        return _exact_cnn(case, seed, device)
    if case["kind"] == "channel":
        return {k: v.cpu().numpy() for k, v in _exact_channel(case, seed, device).items()}
    got = [{k: v.cpu().numpy() for k, v in _exact_channel(c, seed * 1000 + n, device).items()}
           for n, c in enumerate(_sweep_cases(case))]
    if case["uneven"]:
        return {"residual": None, "fields": got}
    return {"residual": None, "fields": {k: np.stack([f[k] for f in got]) for k in FIELDS}}
