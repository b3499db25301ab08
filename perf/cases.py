"""What the framework is timed on: the calls its users make, over the sizes they make them at.

A case of kind
  "step"      builds a ``Solver`` and takes physical steps, then reads the fields (P, S, u) on the
              device: the lattice Boltzmann main path (S refresh, pressure sub-iteration, saturation
              update).  Each pressure solve gets a budget of sweeps (tol = 0, max_sub_iters = the
              budget): the sweep counts that the full runs of the benchmark take, but the same in
              every pass.
  "batch"     advances independent realisations of uneven sizes with one ``Batch``.
  "sweep"     is one ``lbm2p_pressure_sweep_noalloc`` on planes that the caller owns.
  "predict"   is the learned warm start's prediction of the next pressure (features, five 3x3
              convolutions, prediction).
  "train"     is one training step of that operator (forward, backward, Adam).

``exact`` restates the model in 64 bits with plain torch operations on whole arrays.
"""
import ctypes
import math

import numpy as np
import torch

import paper_1808_07554_gb300 as pkg
from paper_1808_07554_gb300.operator import PressureOperator

PERIODIC, NOFLUX, DIRICHLET = 0, 1, 2
QUADRATIC, DECOUPLED, RATIONAL = 0, 1, 2


def _step(name, problem, nx, ny, budget, **kw):
    case = {"name": name, "kind": "step", "problem": problem, "nx": nx, "ny": ny, "budget": budget,
            "steps": 1, "check_every": 8, "warm_start": 0, "storage": 0, "sat_lattice": 9,
            "D_c": 0.0, "mu_n": 2.0, "sigma": 1.0}
    case.update(kw)
    return case


def listed():
    return [
        # one sweep of a caller's own planes, waited for: the smallest call there is
        {"name": "sweep_300x140", "kind": "sweep", "nx": 300, "ny": 140, "walls": "mixed",
         "dense": True},
        # the parity workload: 64 x 64 periodic with dense sources replaced every step
        _step("manufactured_64", "manufactured", 64, 64, 320),
        # Sec. 4.2's example: Dirichlet walls and sources that change every step, S on D2Q5
        _step("dirichlet_128", "dirichlet", 128, 128, 128, sat_lattice=5),
        # a small Monte Carlo realisation with the extrapolated start: several steps per call
        _step("five_spot_256_warm", "five_spot", 256, 256, 24, steps=4, warm_start=1),
        # an odd, ragged lattice with a saturation-dependent diffusivity
        _step("five_spot_1001x603", "five_spot", 1001, 603, 96, check_every=16, D_c=0.5,
              mu_n=5.0),
        # the 1024^2 configuration: a step of a continued solve, and one with the warm start
        _step("five_spot_1024", "five_spot", 1024, 1024, 208, check_every=16),
        _step("five_spot_1024_warm", "five_spot", 1024, 1024, 24, warm_start=1),
        # FP16 storage of the populations, at the loose tolerance it is meant for (few sweeps)
        _step("five_spot_2048_fp16", "five_spot", 2048, 2048, 16, storage=1),
        # the benchmark's default: 4096^2
        _step("five_spot_4096", "five_spot", 4096, 4096, 64, check_every=16),
        # realisations of 128^2 to 1024^2 advanced together, each with its own budget
        {"name": "batch_24", "kind": "batch", "members": 24, "largest": 1024, "budget": 256},
        # the learned warm start at 1024^2, and a training step on 256^2 snapshots
        {"name": "predict_1024", "kind": "predict", "nx": 1024, "ny": 1024},
        {"name": "train_16x256", "kind": "train", "images": 16, "n": 256},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["sweep", "batch", "predict", "train"])
    if kind == "sweep":
        return {"kind": "sweep", "nx": _log_int(rng, 32, 2048), "ny": _log_int(rng, 32, 2048),
                "walls": rng.choice(["noflux", "periodic", "mixed"]),
                "dense": rng.random() < 0.5}
    if kind == "batch":
        return {"kind": "batch", "members": rng.randint(4, 24),
                "largest": rng.choice([256, 512, 1024]), "budget": 16 * rng.randint(2, 16)}
    if kind == "predict":
        return {"kind": "predict", "nx": _log_int(rng, 128, 1024), "ny": _log_int(rng, 128, 1024)}
    if kind == "train":
        return {"kind": "train", "images": rng.randint(1, 16), "n": _log_int(rng, 64, 256)}
    problem = rng.choice(["five_spot"] * 4 + ["manufactured", "dirichlet"])
    every = rng.choice([8, 16])
    warm = int(rng.random() < 0.4)
    lo, hi = (64, 2048) if problem == "five_spot" else (32, 256)
    nx = _log_int(rng, lo, hi)
    ny = nx if rng.random() < 0.4 else max(lo, min(hi, int(nx * rng.uniform(0.5, 1.6))))
    case = _step("", problem, nx, ny,
                 every * (rng.randint(1, 3) if warm else rng.randint(4, 16)),
                 steps=rng.choice([1, 1, 2]), check_every=every, warm_start=warm,
                 storage=int(problem == "five_spot" and rng.random() < 0.1),
                 sat_lattice=rng.choice([9, 9, 5]), mu_n=round(rng.uniform(0.5, 10.0), 3),
                 D_c=rng.choice([0.0, 0.0, 0.3]) if problem == "five_spot" else 0.0,
                 sigma=round(rng.uniform(0.5, 2.0), 3))
    del case["name"]
    return case


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _grf(nx, ny, corr, gen):
    """A standardised Gaussian random field with covariance exp(-r^2 / corr^2), corr in cells."""
    w = torch.randn((ny, nx), generator=gen, device="cuda", dtype=torch.float64)
    ix = torch.arange(nx, device="cuda", dtype=torch.float64)
    iy = torch.arange(ny, device="cuda", dtype=torch.float64)
    dx, dy = torch.minimum(ix, nx - ix), torch.minimum(iy, ny - iy)
    cov = torch.exp(-(dy[:, None] ** 2 + dx[None, :] ** 2) / corr ** 2)
    spec = torch.fft.fft2(cov).real.clamp_min(0.0).sqrt()
    f = torch.fft.ifft2(spec * torch.fft.fft2(w)).real
    return (f - f.mean()) / f.std()


def _nodes(nx, ny, dx):
    x = (torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5) * dx
    y = (torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5) * dx
    return x[None, :].expand(ny, nx), y[:, None].expand(ny, nx)


def _traces(nx, ny, dx, fn):
    """fn(x, y) at the 2n + 1 half-spaced points of each wall."""
    kx = 0.5 * dx * torch.arange(2 * nx + 1, device="cuda", dtype=torch.float64)
    ky = 0.5 * dx * torch.arange(2 * ny + 1, device="cuda", dtype=torch.float64)
    ox, oy = torch.zeros_like(kx), torch.zeros_like(ky)
    return [fn(oy, ky), fn(oy + nx * dx, ky), fn(kx, ox), fn(kx, ox + ny * dx)]


def _problem(c, seed):
    """One problem: parameters, and FP64 arrays on the GPU.  `next` holds the sources and wall
    values of the coming step where these change with time."""
    gen = _gen(seed)
    nx, ny = c["nx"], c["ny"]
    dx = 1.0 / nx
    p = {"nx": nx, "ny": ny, "dx": dx, "phi": 0.2, "mu_w": 1.0, "mu_n": c["mu_n"], "D_s": 0.01,
         "tau_mode": pkg.TAU_REFERENCE, "tau_p": 1.0, "dt": 4.0 * dx * dx,
         "beta": 0.4 if c["sat_lattice"] == 9 else 0.3, "sat_lattice": c["sat_lattice"],
         "D_c": c["D_c"], "mobility": QUADRATIC, "wells": [], "Fp": None, "Fs": None,
         "P_b": None, "S_b": None, "next": None}
    X, Y = _nodes(nx, ny, dx)
    if c["problem"] == "five_spot":
        # wells at opposite corners, no-flux walls; the start is the logarithmic profile of the
        # two wells, so that the pressure relaxes towards the heterogeneous K everywhere
        q = 1e-3
        p["bc"] = (NOFLUX,) * 4
        p["K"] = torch.exp(c["sigma"] * _grf(nx, ny, 16.0, gen))
        p["S0"] = 0.2 + 0.02 * _grf(nx, ny, 12.0, gen)
        r0 = torch.sqrt(X ** 2 + Y ** 2)
        r1 = torch.sqrt((nx * dx - X) ** 2 + (ny * dx - Y) ** 2)
        p["P0"] = 2.0 * q / math.pi * (torch.log(r1) - torch.log(r0)) / (0.04 + 0.64 / c["mu_n"])
        p["wells"] = [(0, 0, q, 0), (nx - 1, ny - 1, q, 1)]
    elif c["problem"] == "manufactured":
        # periodic, dense sources; amplitude and phase from the seed
        ph, amp = torch.rand(2, generator=gen, device="cuda", dtype=torch.float64).tolist()
        a, Lx, Ly = 2.0 * math.pi, nx * dx, ny * dx
        sx, sy = torch.sin(a * X / Lx + ph), torch.sin(a * Y / Ly)
        cy = torch.cos(a * Y / Ly)
        p["bc"] = (PERIODIC,) * 4
        p["K"] = 1.0 + 0.5 * sx * sy
        p["S0"] = 0.5 + 0.25 * sx * sy
        p["P0"] = (0.5 + 0.5 * amp) * sx * cy

        def sources(t):
            Fp = math.exp(-t) * (0.5 + 0.5 * amp) * 30.0 * sx * cy
            Fs = math.exp(-t) * sx * sy
            return Fp - Fp.mean(), Fs

        p["Fp"], p["Fs"] = sources(0.0)
        p["next"] = {"Fp": sources(p["dt"])[0], "Fs": sources(p["dt"])[1]}
    else:
        # Sec. 4.2: P = -cos(pi xi) / (5 pi) - (x + y) / 2, S = sin(pi xi), xi = x + y - 2 t
        pi = math.pi
        t0 = torch.rand(1, generator=gen, device="cuda", dtype=torch.float64).item()
        p.update(phi=1.0, beta=1.0, mobility=RATIONAL, mu_n=1.0, tau_mode=pkg.TAU_PHYSICAL_DT,
                 tau_p=0.0, dt=dx / 10.0, bc=(DIRICHLET,) * 4)

        def P_at(t):
            return lambda x, y: -torch.cos(pi * (x + y - 2.0 * t)) / (5.0 * pi) - 0.5 * (x + y)

        def S_at(t):
            return lambda x, y: torch.sin(pi * (x + y - 2.0 * t))

        def Fs_at(t):
            return 2.0 * pi * pi * 0.01 * torch.sin(pi * (X + Y - 2.0 * t))

        t1 = t0 + p["dt"]
        p["K"] = torch.ones((ny, nx), device="cuda", dtype=torch.float64)
        p["S0"], p["P0"] = S_at(t0)(X, Y), P_at(t0)(X, Y)
        p["Fs"] = Fs_at(t0)
        p["P_b"], p["S_b"] = _traces(nx, ny, dx, P_at(t0)), _traces(nx, ny, dx, S_at(t0))
        p["next"] = {"Fp": None, "Fs": Fs_at(t1), "P_b": _traces(nx, ny, dx, P_at(t1)),
                     "S_b": _traces(nx, ny, dx, S_at(t1))}
    return p


def _host(a):
    if a is None:
        return None
    if isinstance(a, (list, tuple)):
        return [_host(x) for x in a]
    return np.ascontiguousarray(a.cpu().numpy())


INIT_SWEEPS = 32        # sweeps of the t = 0 solve (a fixed count: set-up, not timed)


def _solver(c, p, budget, check_every):
    keys = ("nx", "ny", "dx", "dt", "phi", "beta", "mobility", "mu_w", "mu_n", "D_s", "tau_mode",
            "tau_p", "bc", "wells", "sat_lattice", "D_c")
    return pkg.Solver(K=_host(p["K"]), S0=_host(p["S0"]), P0=_host(p["P0"]), Fp=_host(p["Fp"]),
                      Fs=_host(p["Fs"]), P_b=_host(p["P_b"]), S_b=_host(p["S_b"]), tol=0.0,
                      max_sub_iters=budget, check_every=check_every, init_replay=INIT_SWEEPS,
                      warm_start=c["warm_start"], storage=c["storage"],
                      **{k: p[k] for k in keys})


def _fields_of(sizes):
    """One buffer per field for all lattices, and each lattice's part of it as [ny, nx]."""
    flat = [torch.zeros(sum(nx * ny for nx, ny in sizes), device="cuda") for _ in range(4)]
    views, off = [], 0
    for nx, ny in sizes:
        views.append([f[off:off + nx * ny].view(ny, nx) for f in flat])
        off += nx * ny
    return dict(zip(("P", "S", "ux", "uy"), flat)), views


def _read(solver, out):
    """P, S and the Darcy velocity of the current time level into device tensors."""
    solver.fields_device(out[0], out[1])
    fp = ctypes.POINTER(ctypes.c_float)
    pkg.lbm2p_velocity(solver.h, ctypes.cast(out[2].data_ptr(), fp),
                       ctypes.cast(out[3].data_ptr(), fp), 1)


def _batch_members(c):
    """(size, budget, mu_n, sigma) of each member: sizes uneven as in the batched benchmark, a
    few members with several times the others' sweeps."""
    rng = np.random.default_rng(c["members"])
    sizes = [n for n in (128, 256, 512, 1024) if n <= c["largest"]]
    share = np.array([4.0, 4.0, 4.0, 1.0][:len(sizes)])
    out = []
    for m in range(c["members"]):
        n = int(rng.choice(sizes, p=share / share.sum()))
        if m == 0:
            n = c["largest"]
        b = c["budget"] if rng.random() < 0.25 else max(16, c["budget"] // 64 * 16)
        out.append((n, b, float(rng.uniform(0.5, 10.0)), float(rng.uniform(0.5, 2.0))))
    return out


def _member_case(n, mu_n, sigma):
    return {"problem": "five_spot", "nx": n, "ny": n, "mu_n": mu_n, "sigma": sigma,
            "sat_lattice": 9, "D_c": 0.0, "warm_start": 0, "storage": 0}


def _sweep_inputs(c, seed):
    gen = _gen(seed)
    nx, ny = c["nx"], c["ny"]
    pitch = (nx + 31) // 32 * 32
    bc = {"noflux": (NOFLUX,) * 4, "periodic": (PERIODIC,) * 4,
          "mixed": (NOFLUX, DIRICHLET, PERIODIC, PERIODIC)}[c["walls"]]

    def plane(scale, mean=0.0, k=1):
        t = torch.zeros((k, ny, pitch), device="cuda", dtype=torch.float32)
        t[:, :, :nx] = mean + scale * torch.randn((k, ny, nx), generator=gen, device="cuda")
        return t

    d = {"n_in": plane(1e-3, k=8), "R": plane(1e-2, 0.3)[0], "dP": plane(1e-3)[0],
         "inv_tau": plane(0.0)[0], "Fp": plane(1e-4)[0] if c["dense"] else None, "bc": bc,
         "nx": nx, "ny": ny, "pitch": pitch}
    d["inv_tau"][:, :nx] = 0.4 + 1.2 * torch.rand((ny, nx), generator=gen, device="cuda")
    d["P_b"] = [0.3 + 1e-2 * torch.randn(2 * n + 1, generator=gen, device="cuda")
                if bc[s] == DIRICHLET else None for s, n in enumerate((ny, ny, nx, nx))]
    return d


# channels of the operator's layers, as its users find them in the package
LAYERS = [(16, 32), (32, 32), (32, 32), (32, 32), (32, 16)]


def _weights(gen):
    """One flat FP32 vector in the operator's order: per layer [9][C_out][C_in] and biases."""
    parts = []
    for li, (ci, co) in enumerate(LAYERS):
        w = torch.randn((9, co, ci), generator=gen, device="cuda")
        w *= math.sqrt(2.0 / (9 * (4 if li == 0 else ci)))
        if li == 0:
            w[:, :, 4:] = 0.0
        if li == len(LAYERS) - 1:
            w[:, 1:, :] = 0.0
        parts += [w.reshape(-1), 0.05 * torch.randn(co, generator=gen, device="cuda")]
    return torch.cat(parts)


def _predict_inputs(c, seed):
    gen = _gen(seed)
    nx, ny = c["nx"], c["ny"]
    f32 = lambda a: a.to(torch.float32).contiguous()   # noqa: E731
    S = 0.3 + 0.1 * _grf(nx, ny, 24.0, gen)
    P = 1e-3 * _grf(nx, ny, 48.0, gen)
    return {"lnK": f32(_grf(nx, ny, 16.0, gen)), "S": f32(S),
            "S_prev": f32(S - 1e-4 * _grf(nx, ny, 12.0, gen)), "P": f32(P),
            "P_prev": f32(P - 1e-6 * _grf(nx, ny, 32.0, gen)), "p": _weights(gen)}


def _train_inputs(c, seed):
    gen = _gen(seed)
    k, n = c["images"], c["n"]
    feat = torch.zeros((k, n, n, 16), device="cuda", dtype=torch.bfloat16)
    for i in range(k):
        for ch in range(4):
            feat[i, :, :, ch] = _grf(n, n, 6.0 + 3.0 * ch, gen).to(torch.bfloat16)
    tgt = torch.stack([_grf(n, n, 8.0, gen) for _ in range(k)]).to(torch.float32)
    p = _weights(gen)
    m = 1e-3 * torch.randn(p.shape, generator=gen, device="cuda")
    v = 1e-5 * (0.5 + torch.rand(p.shape, generator=gen, device="cuda"))
    return {"feat": feat, "tgt": tgt.contiguous(), "p": p, "m": m, "v": v}


TRAIN_T = 200           # optimiser steps already taken (a resumed training run)
TRAIN_LR = 1e-3


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        p = _problem(case, seed)
        s = {"kind": kind, "steps": case["steps"], "next": None,
             "solver": _solver(case, p, case["budget"], case["check_every"])}
        s["out"], s["views"] = _fields_of([(p["nx"], p["ny"])])
        if p["next"] is not None:
            s["next"] = {k: _host(v) for k, v in p["next"].items()}
        return s
    if kind == "batch":
        solvers = []
        for m, (n, b, mu_n, sigma) in enumerate(_batch_members(case)):
            c = _member_case(n, mu_n, sigma)
            solvers.append(_solver(c, _problem(c, 1000 * seed + m), b, 16))
        out, views = _fields_of([(s.nx, s.ny) for s in solvers])
        return {"kind": kind, "batch": pkg.Batch(solvers), "solvers": solvers, "out": out,
                "views": views}
    if kind == "sweep":
        d = _sweep_inputs(case, seed)
        d["n_out"] = torch.zeros_like(d["n_in"])
        d["dP_io"] = d["dP"].clone()
        return dict(d, kind=kind)
    op = PressureOperator(seed=1)
    d = _predict_inputs(case, seed) if kind == "predict" else _train_inputs(case, seed)
    op.p.copy_(d["p"])
    op.pb.copy_(d["p"].to(torch.bfloat16))
    if kind == "train":
        op.m.copy_(d["m"])
        op.v.copy_(d["v"])
        op.t = TRAIN_T
        return dict(d, kind=kind, op=op, images=case["images"], n=case["n"])
    ny, nx = d["P"].shape
    d["feat"] = torch.empty((1, ny, nx, 16), device="cuda", dtype=torch.bfloat16)
    d["stats"] = torch.zeros((2, 2), device="cuda", dtype=torch.float64)
    d["P_pred"] = torch.empty_like(d["P"])
    return dict(d, kind=kind, op=op)


# ------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "step":
        solver, nxt = s["solver"], s["next"]
        if nxt is not None:
            solver.set_sources(nxt["Fp"], nxt["Fs"])
            if nxt.get("P_b") is not None:
                for side in range(4):
                    solver.set_dirichlet(side, nxt["P_b"][side], nxt["S_b"][side])
        solver.step(s["steps"])
        _read(solver, s["views"][0])
        return s["out"]
    if kind == "batch":
        s["batch"].step(1)
        for solver, out in zip(s["solvers"], s["views"]):
            _read(solver, out)
        return s["out"]
    if kind == "sweep":
        planes = lambda t: [t[i].data_ptr() for i in range(8)]   # noqa: E731
        r = pkg.lbm2p_pressure_sweep_noalloc(
            s["nx"], s["ny"], s["pitch"], s["bc"], planes(s["n_in"]), planes(s["n_out"]),
            s["R"].data_ptr(), s["inv_tau"].data_ptr(),
            s["Fp"].data_ptr() if s["Fp"] is not None else 0,
            [b.data_ptr() if b is not None else 0 for b in s["P_b"]], s["dP_io"].data_ptr(),
            torch.cuda.current_stream().cuda_stream)
        nx = s["nx"]
        return {"n": s["n_out"][:, :, :nx], "dP": s["dP_io"][:, :nx], "r": r}
    op = s["op"]
    if kind == "predict":
        H, W = s["P"].shape
        st = torch.cuda.current_stream().cuda_stream
        ds, dp = s["stats"][0].data_ptr(), s["stats"][1].data_ptr()
        s["stats"].zero_()
        pkg.lbm2p_op_diff_stats(s["S"].data_ptr(), s["S_prev"].data_ptr(), H * W, ds, st)
        pkg.lbm2p_op_diff_stats(s["P"].data_ptr(), s["P_prev"].data_ptr(), H * W, dp, st)
        pkg.lbm2p_op_features(s["lnK"].data_ptr(), s["S"].data_ptr(), s["S_prev"].data_ptr(),
                              s["P"].data_ptr(), s["P_prev"].data_ptr(), ds, dp,
                              s["feat"].data_ptr(), H, W, 0.2, 0.1, st)
        d = op.forward(s["feat"], 1, H, W)
        pkg.lbm2p_op_predict(s["P"].data_ptr(), s["P_prev"].data_ptr(), d.data_ptr(), dp,
                             s["P_pred"].data_ptr(), H, W, st)
        return {"d": d, "P_pred": s["P_pred"]}
    op.train_step(s["feat"], s["tgt"], s["images"], s["n"], s["n"], lr=TRAIN_LR)
    return {"gradient": op.g, "weights": op.p, "m": op.m, "v": op.v}


# ------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------
# floating-point operations of one node in one pressure sweep: 8 shifted pulls (difference of the
# reference pressure, multiply-add), the sum of Eq. 3-9a, 8 relaxations
SWEEP_FLOPS = 8 * 3 + 8 + 8 * 4
# S refresh, gradient and saturation collision of one node
STEP_FLOPS = 200


def _step_bytes(nodes, dense):
    """State (8 + 9 populations, R, 1/tau_f, S) read and written, K and dense sources read, four
    fields written."""
    return nodes * 4 * (2 * 20 + 1 + dense + 4)


def work(case):
    kind = case["kind"]
    if kind == "step":
        n = case["nx"] * case["ny"]
        dense = {"five_spot": 0, "manufactured": 2, "dirichlet": 1}[case["problem"]]
        return {"bytes": _step_bytes(n, dense),
                "flops": n * case["steps"] * (case["budget"] * SWEEP_FLOPS + STEP_FLOPS)}
    if kind == "batch":
        ms = _batch_members(case)
        return {"bytes": sum(_step_bytes(n * n, 0) for n, _, _, _ in ms),
                "flops": sum(n * n * (b * SWEEP_FLOPS + STEP_FLOPS) for n, b, _, _ in ms)}
    if kind == "sweep":
        n = case["nx"] * case["ny"]
        return {"bytes": n * 4 * (16 + 2 + 2 + int(case["dense"])), "flops": n * SWEEP_FLOPS}
    macs = sum(9 * ci * co for ci, co in LAYERS)
    if kind == "predict":
        n = case["nx"] * case["ny"]
        return {"bytes": n * 4 * 7, "flops": 2 * n * macs}
    n = case["images"] * case["n"] ** 2
    return {"bytes": n * (32 + 4) + 7 * 4 * (macs + sum(co for _, co in LAYERS)),
            "flops": 2 * n * (3 * macs - 9 * LAYERS[0][0] * LAYERS[0][1])}


# ------------------------------------------------------------------------------------------
# the same in 64 bits
# ------------------------------------------------------------------------------------------
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W9 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


def _pull(f, i, bc, trace, wall_weight):
    """Direction i streamed into every node: periodic images, bounce-back, or anti-bounce-back
    with 2 wall_weight x the wall value where the link crosses the wall (corner links use the
    x-side)."""
    ex, ey = EX[i], EY[i]
    out = torch.roll(f[i], (ey, ex), (0, 1))
    ny, nx = out.shape
    if ex and bc[0 if ex > 0 else 1] == PERIODIC:
        ex = 0          # the roll has wrapped it
    if ey and bc[2 if ey > 0 else 3] == PERIODIC:
        ey = 0
    if ey:
        side, row = (2, 0) if ey > 0 else (3, ny - 1)
        own = f[OPP[i]][row]
        if bc[side] == DIRICHLET:
            k = 2 * torch.arange(nx, device=own.device) + 1 - EX[i]
            own = -own + 2.0 * wall_weight * trace[side][k]
        out[row] = own
    if ex:
        side, col = (0, 0) if ex > 0 else (1, nx - 1)
        own = f[OPP[i]][:, col]
        if bc[side] == DIRICHLET:
            k = 2 * torch.arange(ny, device=own.device) + 1 - EY[i]
            own = -own + 2.0 * wall_weight * trace[side][k]
        out[:, col] = own
    return out


def _pull_f(f, p):
    return [None] + [_pull(f, i, p["bc"], p["P_b"], W9[i]) for i in range(1, 9)]


def _mobility(p, S):
    if p["mobility"] == QUADRATIC:
        lw = S * S / p["mu_w"]
        return lw, lw + (1.0 - S) ** 2 / p["mu_n"]
    if p["mobility"] == DECOUPLED:
        return torch.full_like(S, 1.0 / p["mu_w"]), torch.full_like(S, 1.0 / p["mu_w"])
    lt = 1.0 / (0.5 - 0.2 * S)
    return S * lt, lt


def _gradient(a, p, axis):
    """Second-order differences of S0 in lattice units: mirrored at no-flux walls, wrapped when
    periodic, one-sided at Dirichlet walls."""
    lo, hi = (0, 1) if axis == 1 else (2, 3)
    n = a.shape[axis]
    at = lambda j: a.select(axis, j)   # noqa: E731
    up, dn = torch.roll(a, -1, axis), torch.roll(a, 1, axis)
    if p["bc"][lo] != PERIODIC:
        dn.select(axis, 0).copy_(at(0))
        up.select(axis, n - 1).copy_(at(n - 1))
    g = 0.5 * (up - dn)
    if p["bc"][lo] == DIRICHLET:
        g.select(axis, 0).copy_(0.5 * (-3.0 * at(0) + 4.0 * at(1) - at(2)))
    if p["bc"][hi] == DIRICHLET:
        g.select(axis, n - 1).copy_(0.5 * (3.0 * at(n - 1) - 4.0 * at(n - 2) + at(n - 3)))
    return g


class _Model:
    """Sec. 3's two lattice Boltzmann equations on whole FP64 arrays."""

    def __init__(self, p):
        self.p = p
        if p["P_b"] is None:
            p["P_b"] = p["S_b"] = [None] * 4
        dx, dt = p["dx"], p["dt"]
        self.K = p["K"]
        _, lt = _mobility(p, p["S0"])
        if p["tau_mode"] == pkg.TAU_REFERENCE:
            self.s = (p["tau_p"] - 0.5) / (3.0 * torch.log(self.K * lt).mean().exp().item())
        else:
            self.s = dt / dx ** 2
        self.wg = W9 if p["sat_lattice"] == 9 else (1 / 3,) + (1 / 6,) * 4
        if p["sat_lattice"] == 9:
            self.gam = [w * (p["phi"] + (p["beta"] - p["phi"]) *
                             (EX[i] ** 2 + EY[i] ** 2 - 2 / 3) / (2 / 3)) for i, w in enumerate(W9)]
        else:
            self.gam = [(w - (i == 0)) * p["beta"] + (i == 0) * p["phi"]
                        for i, w in enumerate(self.wg)]
        self.q = len(self.wg)
        self.P_prev = None
        f0 = p["P0"]
        self.f = [None] + [w * f0 for w in W9[1:]]
        self.tau = 0.5 + 3.0 * self.s * self.K * lt
        self.solve(INIT_SWEEPS)
        self.init_g()

    def F_p(self):
        F = torch.zeros_like(self.K)
        if self.p["Fp"] is not None:
            F = F + self.s * self.p["dx"] ** 2 * self.p["Fp"]
        for i, j, q, producer in self.p["wells"]:
            F[j, i] += -self.s * q if producer else self.s * q
        return F

    def F_s(self, S):
        F = torch.zeros_like(self.K)
        if self.p["Fs"] is not None:
            F = F + self.p["dt"] * self.p["Fs"]
        lw, lt = _mobility(self.p, S)
        for i, j, q, producer in self.p["wells"]:
            q = self.p["dt"] * q / self.p["dx"] ** 2
            F[j, i] += -q * lw[j, i] / lt[j, i] if producer else q
        return F

    def solve(self, sweeps):
        F = self.F_p() / 8.0
        om = 1.0 / self.tau
        for _ in range(sweeps):
            a = _pull_f(self.f, self.p)
            P = 1.8 * sum(a[1:])
            self.f = [None] + [a[i] + (W9[i] * P - a[i]) * om + F for i in range(1, 9)]

    def pulled(self):
        a = _pull_f(self.f, self.p)
        g = [-3.0 / self.tau * sum(e[i] * a[i] for i in range(1, 9)) for e in (EX, EY)]
        return 1.8 * sum(a[1:]), g

    def tau_g(self, S):
        p = self.p
        lw, lt = _mobility(p, S)
        D = p["D_s"] + p["D_c"] * self.K * lw * (lt - lw) / lt
        return 0.5 + 3.0 * D * p["dt"] / (p["beta"] * p["dx"] ** 2), lw

    def collide_g(self, q, S, Fs, g):
        tg, lw = self.tau_g(S)
        gam = -3.0 * self.p["dt"] / self.p["dx"] ** 2 * lw * self.K
        self.g = [q[i] + (self.gam[i] * S - q[i]) / tg + self.wg[i] * (1 - 0.5 / tg) * Fs +
                  gam * self.wg[i] * (EX[i] * g[0] + EY[i] * g[1]) / tg for i in range(self.q)]
        self.S = S

    def init_g(self):
        p, S0 = self.p, self.p["S0"]
        _, g = self.pulled()
        sx, sy = _gradient(S0, p, 1), _gradient(S0, p, 0)
        Fs = self.F_s(S0)
        tg, lw = self.tau_g(S0)
        gam = -3.0 * p["dt"] / p["dx"] ** 2 * lw * self.K
        q = []
        for i in range(self.q):
            w, G = self.wg[i], self.gam[i]
            neq = -tg * ((G / p["phi"] - w * (1 - 0.5 / tg)) * Fs + G * (EX[i] * sx + EY[i] * sy) -
                         gam * w * (EX[i] * g[0] + EY[i] * g[1]) / tg)
            q.append(G * S0 + neq)
        self.collide_g(q, (sum(q) + 0.5 * Fs) / p["phi"], Fs, g)

    def stream_g(self):
        p = self.p
        q = [self.g[0]] + [_pull(self.g, i, p["bc"], p["S_b"], self.gam[i])
                           for i in range(1, self.q)]
        s = sum(q)
        Fs = self.F_s(s / p["phi"])
        return q, (s + 0.5 * Fs) / p["phi"], Fs

    def step(self, sweeps, warm):
        _, S, _ = self.stream_g()
        if warm:
            P, _ = self.pulled()
            if self.P_prev is not None:
                self.f = [None] + [self.f[i] + W9[i] * (P - self.P_prev) for i in range(1, 9)]
            self.P_prev = P
        self.tau = 0.5 + 3.0 * self.s * self.K * _mobility(self.p, S)[1]
        self.solve(sweeps)
        _, g = self.pulled()
        q, S, Fs = self.stream_g()
        self.collide_g(q, S, Fs, g)

    def fields(self):
        P, g = self.pulled()
        kl = self.K * _mobility(self.p, self.S)[1] / self.p["dx"]
        return {"P": P, "S": self.S, "ux": -kl * g[0], "uy": -kl * g[1]}


def _exact_step(c, seed, steps, budget):
    p = _problem(c, seed)
    m = _Model(p)
    if p["next"] is not None:
        p.update(p["next"])
    for _ in range(steps):
        m.step(budget, c["warm_start"])
    return m.fields()


def _exact_sweep(c, seed):
    d = _sweep_inputs(c, seed)
    nx = d["nx"]
    up = lambda t: t[..., :nx].double()   # noqa: E731
    n, R, om = up(d["n_in"]), up(d["R"]), 1.0 * up(d["inv_tau"])
    f = [None] + [n[i - 1] + W9[i] * R for i in range(1, 9)]
    trace = [b.double() if b is not None else None for b in d["P_b"]]
    a = _pull_f(f, {"bc": d["bc"], "P_b": trace})
    P = 1.8 * sum(a[1:])
    F = up(d["Fp"]) / 8.0 if d["Fp"] is not None else 0.0
    out = torch.stack([a[i] + (W9[i] * P - a[i]) * om + F - W9[i] * R for i in range(1, 9)])
    dP = P - R
    e, u = dP - up(d["dP"]), P
    r = ((e - e.mean()).square().sum() / (u - u.mean()).square().sum()).sqrt()
    return {"n": out, "dP": dP, "r": r.item()}


def _layers(p):
    off = 0
    for ci, co in LAYERS:
        w = p[off:off + 9 * ci * co].reshape(3, 3, co, ci).permute(2, 3, 0, 1)
        b = p[off + 9 * ci * co:off + 9 * ci * co + co]
        off += 9 * ci * co + co
        yield w, b


def _network(x, p):
    """x [n, 16, H, W] through the five convolutions; channel 0 of the last."""
    ws = list(_layers(p))
    for li, (w, b) in enumerate(ws):
        x = torch.nn.functional.conv2d(x, w, b, padding=1)
        if li + 1 < len(ws):
            x = torch.relu(x)
    return x[:, 0]


def _bf16_weights(p):
    """The convolutions read BF16 weights and FP32 biases."""
    q = p.to(torch.bfloat16).double()
    off = 0
    for ci, co in LAYERS:
        off += 9 * ci * co
        q[off:off + co] = p[off:off + co].double()
        off += co
    return q


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        # FP16 storage rounds every sweep: its error against 64 bits is the storage's own
        got = _exact_step(case, seed, case["steps"], case["budget"])
        return {k: v.reshape(-1) for k, v in got.items()}
    if kind == "batch":
        got = [_exact_step(_member_case(n, mu_n, sigma), 1000 * seed + m, 1, b)
               for m, (n, b, mu_n, sigma) in enumerate(_batch_members(case))]
        return {k: torch.cat([g[k].reshape(-1) for g in got]) for k in got[0]}
    if kind == "sweep":
        return _exact_sweep(case, seed)
    if kind == "predict":
        d = {k: v.double() if k != "p" else v for k, v in _predict_inputs(case, seed).items()}
        dS, dP = d["S"] - d["S_prev"], d["P"] - d["P_prev"]
        sd = lambda a: a.std(correction=0)   # noqa: E731
        feat = torch.zeros((1, 16) + tuple(d["P"].shape), device="cuda", dtype=torch.float64)
        feat[0, 0], feat[0, 1] = d["lnK"], (d["S"] - 0.2) / 0.1
        feat[0, 2], feat[0, 3] = dS / sd(dS), dP / sd(dP)
        y = _network(feat, _bf16_weights(d["p"]))
        return {"d": y, "P_pred": 2.0 * d["P"] - d["P_prev"] + sd(dP) * y[0]}
    d = _train_inputs(case, seed)
    p = _bf16_weights(d["p"]).requires_grad_(True)
    y = _network(d["feat"].double().permute(0, 3, 1, 2).contiguous(), p)
    (y - d["tgt"].double()).square().mean().backward()
    g = p.grad.clone()
    m = 0.9 * d["m"].double() + 0.1 * g
    v = 0.999 * d["v"].double() + 0.001 * g * g
    t = TRAIN_T + 1
    step = (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return {"gradient": g, "weights": d["p"].double() - TRAIN_LR * step, "m": m, "v": v}
