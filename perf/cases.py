"""The work that users of this package have it do, as cases to time.

Four kinds, each through the package's public entry points:

  solve    one solver instance: a whole run from the equilibrium start
           (``Solver.reset``, ``run``, ``observables``, ``trace``) and the
           state of both grids at its end (``get_state``), as a program does
           that keeps a checkpoint
  sweep    ``batch_run`` over points of the sweep box with the package's grid
           rule (``workloads.sweep_grid_rule``)
  train    a part of an epoch of ``Surrogate.train``: Adam steps over given
           minibatches, and the updated weights (``get_params``)
  predict  ensemble inference, of host arrays (``predict``) or of device
           arrays (``predict_device``)

The runs are shortened (the configured ones have 20 to 50 drive periods); the
grids, time steps and launch options are the configured ones.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1401_6047_gb300 import bte
from paper_1401_6047_gb300 import surrogate as S
from paper_1401_6047_gb300 import workloads as W

# operations of one cell-update (both half-steps of one cell; a multiply-add
# counts two) in the form of the update with the fewest operations
FLOPS_PER_CELL = 66
PARAMS = 133634  # of one ensemble member
FLOPS_PER_POINT = 2 * PARAMS  # of one member's forward pass


def listed():
    return [
        # the smallest call: a few steps of the plain configuration, where
        # launches and latency count
        dict(name="point_fp64_few", kind="solve", base="c1", n_max=30, m_points=201, fp64=True, mode=0,
             steps=32, b_omega=0.0),
        # the plain configuration for one drive period
        dict(name="point_fp64", kind="solve", base="c1", n_max=30, m_points=201, fp64=True, mode=0,
             steps=6283, b_omega=0.0),
        # the same grid in the mode the package offers for small grids
        dict(name="point_fp64_on_chip", kind="solve", base="c1", n_max=30, m_points=201, fp64=True, mode=3,
             steps=6283, b_omega=0.0),
        # a ragged middle-sized grid in a time-dependent field
        dict(name="mid_fp32_bfield", kind="solve", base="c2", n_max=137, m_points=1533, fp64=False, mode=0,
             steps=2001, b_omega=0.3),
        # 401 x 4001: one drive period in mixed precision, and the FP64 run
        # that its error is stated against
        dict(name="large_fp32", kind="solve", base="c2", n_max=400, m_points=4001, fp64=False, mode=0,
             steps=6283, b_omega=0.0),
        dict(name="large_fp64", kind="solve", base="c2", n_max=400, m_points=4001, fp64=True, mode=0,
             steps=400, b_omega=0.0),
        # 2049 x 8193: the low-temperature run, larger than any cache
        dict(name="lowtemp_fp32", kind="solve", base="c3", n_max=2048, m_points=8193, fp64=False, mode=0,
             steps=4096, b_omega=0.0),
        # the run timed in the paper's Table 1: few harmonics, wide grid
        dict(name="table1_fp32", kind="solve", base="table1", n_max=119, m_points=4000, fp64=False, mode=0,
             steps=6283, b_omega=0.0),
        # a slice of the 4096-point sweep, each point for one drive period
        dict(name="sweep_fp32", kind="sweep", points=256, fp64=False, periods=1.0, grid_seed=1401),
        # a few points in FP64, as one checks a sweep
        dict(name="sweep_fp64", kind="sweep", points=12, fp64=True, periods=0.125, grid_seed=2014),
        # training of the 8-member ensemble with the shipped batch size
        dict(name="train", kind="train", members=8, batch=1024, steps=32, data=20000),
        # inference of the whole point set on the device
        dict(name="predict_device", kind="predict", members=8, points=1000000, device=True),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["solve"] * 6 + ["sweep"] * 2 + ["train", "predict", "predict"])
    if kind == "solve":
        fp64 = rng.random() < 0.35
        mode = 3 if rng.random() < 0.15 else 0
        b_omega = rng.choice([0.0, 0.0, round(rng.uniform(0.05, 0.5), 3)])
        if mode == 3:  # small grids only
            n_max, m_points = rng.randint(16, 47), rng.randint(96, 256)
        else:
            n_max, m_points = log_int(20, 2048), log_int(128, 8193)
        cells = (n_max + 1) * m_points
        # a pass of up to about half a second, the largest with the most
        # cell-updates; small grids for up to one drive period
        steps = int(min((1.2e9 if fp64 else 3e10) / cells, 6283) * rng.uniform(0.3, 1.0))
        return dict(kind="solve", base="c2", n_max=n_max, m_points=m_points, fp64=fp64, mode=mode,
                    steps=max(steps, 16), b_omega=b_omega)
    if kind == "sweep":
        fp64 = rng.random() < 0.3
        points = log_int(4, 16) if fp64 else log_int(8, 256)
        return dict(kind="sweep", points=points, fp64=fp64,
                    periods=round(rng.uniform(0.05, 0.125) if fp64 else rng.uniform(0.3, 1.0), 3),
                    grid_seed=rng.randint(0, 10**6))
    if kind == "train":
        return dict(kind="train", members=rng.choice([1, 4, 8, 8]), batch=log_int(100, 4096),
                    steps=rng.randint(8, 40), data=log_int(5000, 200000))
    device = rng.random() < 0.5
    return dict(kind="predict", members=rng.choice([1, 4, 8, 8]), points=log_int(100, 1000000), device=device)


# --- solver parameters ------------------------------------------------------

def _solve_params(case, seed):
    """The configuration's drive, field and temperature, a few per cent off
    by the seed, on the case's grid and run length (the second half of the
    run averaged)."""
    base = {"c1": W.c1_fp64, "c2": W.c2, "c3": W.c3, "table1": W.paper_table1}[case["base"]]()
    r = np.random.default_rng([seed, 7])
    f = 1.0 + 0.05 * r.uniform(-1.0, 1.0, size=4)
    period = round(2.0 * math.pi / (base.omega * base.dt))
    # spacing of the configured grid, so that a smaller grid covers a smaller range
    half = 0.5 * (base.phiy_max - base.phiy_min) * (case["m_points"] - 1) / (base.m_points - 1)
    half = max(half, 7.0 / math.sqrt(base.mu) + 1.5 * (base.B + case["b_omega"]))  # the sweep's range
    return base.replace(E_dc=base.E_dc * f[0], E_omega=base.E_omega * f[1], B=base.B * f[2], mu=base.mu * f[3],
                        n_max=case["n_max"], m_points=case["m_points"], phiy_min=-half, phiy_max=half,
                        periods=case["steps"] / period, avg_window=0.5 * case["steps"] / period,
                        precision=W.FP64 if case["fp64"] else W.FP32_MIXED,
                        B_omega=case["b_omega"], B_phase=0.5 if case["b_omega"] else 0.0)


def _sweep_params(case, seed):
    """Temperatures, fields and frequencies (so grids and run lengths) by the
    case, drives by the seed; the last half of each run averaged."""
    pts = W.sweep_points(case["points"], seed=case["grid_seed"], periods=case["periods"],
                         avg_window=0.5 * case["periods"], precision=W.FP64 if case["fp64"] else W.FP32_MIXED)
    x = W.sweep_matrix(case["points"], seed)
    return [p.replace(E_dc=float(x[i, 0]), E_omega=float(x[i, 1])) for i, p in enumerate(pts)]


def _nearest(x):
    return math.floor(x + 0.5)


def _steps_of(p):
    return _nearest(p.periods * _nearest(2.0 * math.pi / (p.omega * p.dt)))


# --- surrogate inputs ---------------------------------------------------------

Y_MEAN, Y_STD = (0.02, 0.25), (0.15, 0.12)


def _weights(case, seed):
    return S.init_params(case["members"], seed=1000 * (seed % 100000))


def _train_set(case, seed):
    x = W.sweep_matrix(case["data"], seed).astype(np.float32)
    # smooth targets of the size of the solver's absorption and drift velocity
    e, eo, om, b, mu = x.T.astype(np.float64)
    y = np.stack([0.3 * np.cos(e / om) * np.exp(-0.2 * b) + 0.05 * eo, e / (1.0 + e * e) * np.tanh(0.5 * mu)], axis=1)
    r = np.random.default_rng([seed, 3])
    order = r.integers(0, case["data"], size=(case["steps"], case["members"], case["batch"]), dtype=np.int32)
    t = (np.arange(case["steps"]) + 0.5) / 4000.0
    lr = (2e-5 + 0.5 * (2e-3 - 2e-5) * (1.0 + np.cos(np.pi * t))).astype(np.float32)
    return x, y.astype(np.float32), order, lr


# --- preparation and the timed pass -------------------------------------------

def prepare(case, seed):
    if case["kind"] == "solve":
        return {"case": case, "solver": bte.Solver(_solve_params(case, seed), resident=case["mode"])}
    if case["kind"] == "sweep":
        return {"case": case, "points": _sweep_params(case, seed)}
    if case["kind"] == "train":
        x, y, order, lr = _train_set(case, seed)
        sur = S.Surrogate(Y_MEAN, Y_STD, members=case["members"], batch_capacity=4096)
        sur.set_data(x, y)
        return {"case": case, "sur": sur, "start": _weights(case, seed), "order": order, "lr": lr}
    stream = torch.cuda.Stream()
    sur = S.Surrogate(Y_MEAN, Y_STD, members=case["members"], batch_capacity=65536, stream=stream.cuda_stream)
    sur.set_params(_weights(case, seed))
    n = case["points"]
    x = W.sweep_matrix(n, seed).astype(np.float32)
    state = {"case": case, "sur": sur, "x": x, "stream": stream}
    if case["device"]:
        state["x"] = torch.from_numpy(x).cuda()
        state["mean"] = torch.empty(n, 2, device="cuda")
        state["std"] = torch.empty(n, 2, device="cuda")
        state["mask"] = torch.empty(n, dtype=torch.uint8, device="cuda")
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "solve":
        s = state["solver"]
        s.reset()
        s.run()
        o = s.observables()
        v, norm = s.trace()
        aw, bw = s.get_state(0)
        af, bf = s.get_state(1)
        return {"v_dr": o.v_dr, "norm": o.norm, "v_dc_avg": o.v_dc_avg, "absorption": o.absorption, "steps": o.step,
                "trace_v": v, "trace_norm": norm, "a_whole": aw, "b_whole": bw, "a_frac": af, "b_frac": bf}
    if case["kind"] == "sweep":
        res = bte.batch_run(state["points"])
        return {k: np.array([getattr(o, k) for o in res])
                for k in ("v_dr", "norm", "v_dc_avg", "absorption", "step", "status")}
    if case["kind"] == "train":
        state["sur"].set_params(state["start"])
        loss = state["sur"].train(state["order"], state["lr"])
        return {"params": state["sur"].get_params(), "loss": loss}
    if not case["device"]:
        mean, std, mask = state["sur"].predict(state["x"])
        return {"mean": mean, "std": std, "mask": mask.astype(np.uint8)}
    state["sur"].predict_device(state["x"].data_ptr(), case["points"], state["mean"].data_ptr(),
                                state["std"].data_ptr(), state["mask"].data_ptr())
    return {"mean": state["mean"], "std": state["std"], "mask": state["mask"]}


def work(case):
    if case["kind"] == "solve":
        elem = 8 if case["fp64"] else 4
        cells = (case["n_max"] + 1) * case["m_points"]
        # the state at the end and the trace are written once
        return {"bytes": 4 * elem * cells + 16 * case["steps"], "flops": FLOPS_PER_CELL * cells * case["steps"]}
    if case["kind"] == "sweep":
        pts = _sweep_params(case, 0)
        return {"bytes": sum(2 * 4 * (8 if case["fp64"] else 4) * (p.n_max + 1) for p in pts),
                "flops": sum(FLOPS_PER_CELL * p.cells * _steps_of(p) for p in pts)}
    if case["kind"] == "train":
        m, b = case["members"], case["batch"]
        # per step: the weights and both moments read and written, the
        # minibatch read; a forward and two backward products
        return {"bytes": case["steps"] * m * (6 * 4 * PARAMS + b * 32), "flops": case["steps"] * m * b * 3 * FLOPS_PER_POINT}
    n, m = case["points"], case["members"]
    return {"bytes": n * (20 + 17) + 4 * m * PARAMS, "flops": n * m * FLOPS_PER_POINT}


# --- the same in 64 bits ----------------------------------------------------------

def _exact_solve(p, steps):
    """The scheme in complex form, z = a + i b: T solves (nu - i th1) z' =
    (xi + i th) z + S + h a0 with S = c (D b_{n+1} - D b_{n-1}) + i c (chi D
    a_{n-1} - D a_{n+1}), D the central phi_y difference."""
    dev = "cuda"
    N1, M1 = p.n_max + 1, p.m_points
    f8 = dict(dtype=torch.float64, device=dev)
    per = _nearest(2.0 * math.pi / (p.omega * p.dt))
    dt = 2.0 * math.pi / (p.omega * per)
    dphi = (p.phiy_max - p.phiy_min) / (M1 - 1)
    phi = p.phiy_min + dphi * torch.arange(M1, **f8)
    n = torch.arange(N1, **f8)[:, None]
    # I_n / I_0 from the Fourier integral of exp(mu cos x)
    q = max(4096, 4 * N1)
    w = np.exp(p.mu * (np.cos(2.0 * np.pi * np.arange(q) / q) - 1.0))
    ratio = np.real(np.fft.rfft(w))[:N1] / np.sum(w)
    sigma = np.ones(N1)
    sigma[0] = 0.5
    a0 = torch.from_numpy(sigma * ratio / math.pi).to(dev)[:, None] * (
        math.sqrt(p.mu / (2.0 * math.pi * p.alpha)) * torch.exp(-0.5 * p.mu * phi * phi))[None, :]
    chi = torch.ones(N1, 1, **f8)
    chi[1] = 2.0
    chi[0] = 0.0

    def E(t):
        return p.E_dc + p.E_omega * math.cos(p.omega * t)

    def B(t):
        return p.B + p.B_omega * math.cos(p.omega * t + p.B_phase)

    def diff(x):
        d = torch.zeros_like(x)
        d[:, 1:] += x[:, :-1].neg()
        d[:, :-1] += x[:, 1:]
        return d

    def advance(z, src, t, h, t_src):
        """T over a step h from t, the stencil taken from src at time t_src."""
        a, b = z
        c = B(t_src) * h / (4.0 * dphi)
        da, db = diff(src[0]), diff(src[1])
        g = a0 * h
        g[:-1].add_(db[1:], alpha=c)
        g[1:].sub_(db[:-1], alpha=c)
        s = torch.zeros_like(a)
        s[1:] += c * chi[1:] * da[:-1]
        s[:-1].sub_(da[1:], alpha=c)
        nu, xi = 1.0 + 0.5 * h, 1.0 - 0.5 * h
        th = n * ((E(t) + B(t) * phi) * (0.5 * h))[None, :]
        th1 = n * ((E(t + h) + B(t + h) * phi) * (0.5 * h))[None, :]
        g.add_(a, alpha=xi).sub_(b * th)
        s.add_(b, alpha=xi).add_(a * th)
        inv = 1.0 / (nu * nu + th1 * th1)
        an = (nu * g - s * th1) * inv
        bn = (g * th1 + nu * s) * inv
        bn[0] = 0.0
        return an, bn

    whole = (a0.clone(), torch.zeros_like(a0))
    frac = advance(whole, whole, 0.0, 0.5 * dt, 0.0)
    v, norm = torch.empty(steps + 1, **f8), torch.empty(steps + 1, **f8)
    sq = math.sqrt(p.alpha)
    for k in range(steps + 1):
        v[k] = math.pi * sq * dphi * whole[1][1].sum()
        norm[k] = 2.0 * math.pi * sq * dphi * whole[0][0].sum()
        if k == steps:
            break
        t = k * dt
        whole = advance(whole, frac, t, dt, t + 0.5 * dt)
        frac = advance(frac, whole, t + 0.5 * dt, dt, t + dt)
    kw = max(1, _nearest(p.avg_window * per))
    last = v[steps - kw + 1:]
    ph = 2.0 * math.pi * ((steps - kw + 1 + torch.arange(kw, **f8)) % per) / per
    return {"v_dr": v[-1].item(), "norm": norm[-1].item(), "v_dc_avg": last.mean().item(),
            "absorption": 2.0 / ratio[1] * (last * torch.cos(ph)).mean().item(),
            "trace_v": v, "trace_norm": norm, "a_whole": whole[0], "b_whole": whole[1],
            "a_frac": frac[0], "b_frac": frac[1]}


def _net(w, x):
    """Forward pass of all members [m, ...] over x [m or 1, n, 5]; weights as
    a list of tensors."""
    h = x
    for k in range(3):
        z = h @ w[2 * k].transpose(1, 2) + w[2 * k + 1][:, None, :]
        h = z * torch.sigmoid(z)
    return h @ w[6].transpose(1, 2) + w[7][:, None, :]


def _unpack(p):
    out, o = [], 0
    for shape in ((256, 5), (256,), (256, 256), (256,), (256, 256), (256,), (2, 256), (2,)):
        k = int(np.prod(shape))
        out.append(p[:, o:o + k].reshape((p.shape[0],) + shape))
        o += k
    return out


def _box(x):
    lo = torch.tensor([v[0] for v in W.SWEEP_BOX.values()], dtype=torch.float64, device="cuda")
    hi = torch.tensor([v[1] for v in W.SWEEP_BOX.values()], dtype=torch.float64, device="cuda")
    return 2.0 * (x - lo) / (hi - lo) - 1.0


def exact(case, seed):
    mean = torch.tensor(Y_MEAN, dtype=torch.float64, device="cuda")
    std = torch.tensor(Y_STD, dtype=torch.float64, device="cuda")
    if case["kind"] == "solve":
        p = _solve_params(case, seed)
        # about 40 passes over a 64-bit array each step
        if case["steps"] * (4e-4 + 40 * 16.0 * p.cells / 5e12) > 18.0:
            return None
        out = _exact_solve(p, case["steps"])
        out["steps"] = None
        return out
    if case["kind"] == "sweep":
        pts = _sweep_params(case, seed)
        if sum(_steps_of(p) * (4e-4 + 40 * 16.0 * p.cells / 5e12) for p in pts) > 18.0:
            return None
        res = [_exact_solve(p, _steps_of(p)) for p in pts]
        out = {k: np.array([r[k] for r in res]) for k in ("v_dr", "norm", "v_dc_avg", "absorption")}
        out["step"] = out["status"] = None
        return out
    w0 = torch.from_numpy(_weights(case, seed)).cuda().double()
    if case["kind"] == "train":
        x, y, order, lr = (torch.from_numpy(v).cuda() for v in _train_set(case, seed))
        xs, ys = _box(x.double()), (y.double() - mean) / std
        p = w0.clone().requires_grad_(True)
        m, v, losses = torch.zeros_like(w0), torch.zeros_like(w0), []
        for s in range(case["steps"]):
            idx = order[s].long()
            loss = 0.5 * ((_net(_unpack(p), xs[idx]) - ys[idx]) ** 2).sum(dim=(1, 2)) / case["batch"]
            losses.append(loss.detach())
            (g,) = torch.autograd.grad(loss.sum(), p)
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            step = float(lr[s]) * (m / (1 - 0.9 ** (s + 1))) / ((v / (1 - 0.999 ** (s + 1))).sqrt() + 1e-8)
            p = (p.detach() - step).requires_grad_(True)
        return {"params": p.detach(), "loss": torch.stack(losses)}
    x = _box(torch.from_numpy(W.sweep_matrix(case["points"], seed).astype(np.float32)).cuda().double())
    w, means, stds = _unpack(w0), [], []
    for part in x.split(32768):
        yy = _net(w, part[None].expand(case["members"], -1, -1)) * std + mean
        means.append(yy.mean(dim=0))
        stds.append(yy.std(dim=0, correction=0))
    # one member has no spread
    return {"mean": torch.cat(means), "std": torch.cat(stds) if case["members"] > 1 else None, "mask": None}
