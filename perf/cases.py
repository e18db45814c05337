"""What this framework is measured on: its solver and its warm-start network
over the range of their use, through the entry points a program calls.

Kinds of cases
  flow     one lattice: initial state, `steps` time steps in one call, density
           and velocity read into device arrays (lb_init, lb_step, lb_moments;
           FP64 handles also the global sums of lb_reduce_async, the check a
           reference run makes).
  monitor  the same between host arrays, the way a production run is driven:
           initial density and results in page-locked memory, every step's
           record written into a page-locked ring.
  batch    an ensemble of independent lattices of uneven sizes stepped together
           (lb_batch_*), each started and read on its own.
  train    one optimiser step of the network: forward, backward, Adam, gradients
           and weights read back.
  predict  a warm start: the network's prediction turned into initial fields on
           the device, a solver started from them and read.

The lattices, temperatures, force amplitudes, wavelengths, wall speeds,
relaxation times and stencils are those of this repository's workloads, paper
regimes and tests (paper_1307_6703_gb300/workloads.py, regimes.py,
warmstart.py): a = 3/8, b = 1/3, kappa = 0.1, N = 0.3, Q = 2.0.
"""
import math

import numpy as np
import torch

import paper_1307_6703_gb300 as lbm
from paper_1307_6703_gb300 import fno as fno_mod

A_VDW, B_VDW, KAPPA, ST_N, ST_Q = 3.0 / 8.0, 1.0 / 3.0, 0.1, 0.3, 2.0
T_C = 1.0 / 3.0
NOISE = 0.01 / 3.5                       # noisy uniform start around the critical density 1
PREC = {"fp64": lbm.LB_FP64, "fp32": lbm.LB_FP32, "bf16": lbm.LB_BF16DEV, "fp16": lbm.LB_FP16DEV}
SITE_BYTES = {"fp64": 72, "fp32": 36, "bf16": 20, "fp16": 20}
SCALES = (0.5, 0.05, 0.05)               # network outputs: (n - 1) / 0.5, u_x / 0.05, u_y / 0.05
WIDTH, HIDDEN, LAYERS, MX, MY, OUT = 32, 64, 4, 16, 8, 3
LR = 2e-3


def _flow(name, prec, nx, ny, steps, *, walls=True, uw=0.05, a0=1e-4, lam=64.0, tr=0.95, tau=1.0, start="noise",
          tune=False, kind="flow"):
    return {"name": name, "kind": kind, "prec": prec, "nx": nx, "ny": ny, "steps": steps, "walls": walls, "uw": uw,
            "a0": a0, "lam": lam, "tr": tr, "tau": tau, "start": start, "tune": tune}


def listed():
    return [
        # One step of the smallest lattice of the test problems, read after it: a
        # program that couples to the solver step by step.  Launches and latency.
        _flow("fp32_64x32_one_step", "fp32", 64, 32, 1, uw=0.0, a0=1e-3, lam=32.0),
        # The sheared channel of the parity and wave-statistics runs: a lattice that
        # leaves most of the GPU idle unless it is cut finely.
        _flow("fp32_512x256", "fp32", 512, 256, 100, lam=128.0),
        # The headline lattice, tuned once as a long run does.
        _flow("fp32_4096x1024", "fp32", 4096, 1024, 20, lam=512.0, tune=True),
        # The same lattice in 16-bit deviation storage, and a periodic one in the other
        # format at the paper's larger relaxation time, from a developed state.
        _flow("bf16_4096x1024", "bf16", 4096, 1024, 20, lam=512.0, tune=True),
        _flow("fp16_2048x512_periodic", "fp16", 2048, 512, 20, walls=False, uw=0.0, tau=2.0, start="stripes"),
        # Odd sizes (the general FP32 kernel): droplet and channel studies on sizes
        # that are not multiples of 4.
        _flow("fp32_1021x509_ragged", "fp32", 1021, 509, 20, tau=2.0, start="stripes"),
        # The double-precision path that the error of every other format is measured against.
        _flow("fp64_512x256", "fp64", 512, 256, 20, lam=128.0),
        # 64 uneven lattices of a parameter sweep.
        {"name": "batch_fp32_64", "kind": "batch", "prec": "fp32", "count": 64, "steps": 50, "nx_max": 1024,
         "ny_max": 256},
        # The headline lattice driven from and to host memory, monitored at every step.
        _flow("monitored_fp32_4096x1024", "fp32", 4096, 1024, 20, lam=512.0, tune=True, kind="monitor"),
        # Training of the warm-start network at its two training sizes.
        {"name": "train_16x256x64", "kind": "train", "batch": 16, "nx": 256, "ny": 64},
        {"name": "train_8x512x128", "kind": "train", "batch": 8, "nx": 512, "ny": 128},
        # Warm start of the largest warm-started lattice.
        {"name": "predict_2048x512", "kind": "predict", "batch": 1, "nx": 2048, "ny": 512},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _physics(rng):
    return {"a0": rng.uniform(1e-4, 5e-4), "lam": rng.choice([32.0, 64.0]), "tr": rng.uniform(0.92, 0.96),
            "tau": rng.choice([1.0, 1.0, 2.0, 3.0])}


def draw(rng):
    kind = rng.choice(["flow"] * 6 + ["monitor", "batch", "train", "train", "predict"])
    if kind in ("flow", "monitor"):
        prec = rng.choice(["fp32", "fp32", "bf16", "fp16", "fp64"]) if kind == "flow" else "fp32"
        ragged = prec == "fp64" or (prec == "fp32" and kind == "flow" and rng.random() < 0.3)
        q = 1 if ragged else (8 if prec in ("bf16", "fp16") else 4)
        top = 1024 if ragged else 4096
        nx = max(16, q * round(_log(rng, 32, top) / q))
        ny = round(_log(rng, 24, 512 if ragged else 1024))
        walls = rng.random() < 0.7
        # enough steps for a run, fewer on the larger lattices
        steps = max(1, min(100, round(_log(rng, 1, 100)), 20 * 4096 * 1024 // (nx * ny)))
        if prec == "fp64":
            steps = max(1, min(steps, 20 * 512 * 256 // (nx * ny)))
        return {"kind": kind, "prec": prec, "nx": nx, "ny": ny, "steps": steps, "walls": walls,
                "uw": rng.uniform(0.0, 0.1) if walls else 0.0, "start": rng.choice(["noise", "stripes"]),
                "tune": False, **_physics(rng)}
    if kind == "batch":
        return {"kind": "batch", "prec": rng.choice(["fp32", "bf16"]), "count": round(_log(rng, 4, 64)),
                "steps": 2 * rng.randint(5, 25), "nx_max": rng.choice([256, 512, 1024]), "ny_max": rng.choice([128, 256])}
    if kind == "train":
        nx, ny = 8 * rng.randint(8, 64), rng.randint(32, 128)
        return {"kind": "train", "batch": max(1, min(rng.randint(1, 16), 8 * 512 * 128 // (nx * ny))), "nx": nx, "ny": ny}
    return {"kind": "predict", "batch": rng.randint(1, 2), "nx": 8 * round(_log(rng, 16, 256)), "ny": round(_log(rng, 64, 512))}


# ------------------------------------------------------------------ inputs

def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed):
    return np.random.default_rng(int(seed))


def _stripes(c, seed):
    """A developed state: a wavy liquid slab between vapour, sheared between the
    walls, with the small-scale disturbance of a running simulation.  FP64 fields
    (n, u_x) on the device."""
    g, dev = _gen(seed), _dev()
    x = torch.arange(c["nx"], dtype=torch.float64, device=dev)[None, :]
    y = torch.arange(c["ny"], dtype=torch.float64, device=dev)[:, None]
    nx, ny = c["nx"], c["ny"]
    wave = sum(float(a) * torch.cos(2.0 * math.pi * k * x / nx + float(p))
               for k, a, p in zip((1, 2, 3), g.uniform(0.3, 1.0, 3), g.uniform(0.0, 6.2, 3)))
    n = 1.0 + 0.4 * (torch.tanh((y - ny / 4 - wave) / 4.0) - torch.tanh((y - 3 * ny / 4 + wave) / 4.0) - 1.0)
    tg = torch.Generator(device=dev)
    tg.manual_seed(int(seed))
    n = n + 1e-3 * (2.0 * torch.rand((ny, nx), dtype=torch.float64, device=dev, generator=tg) - 1.0)
    u = c["uw"] * (2.0 * y / (ny - 1) - 1.0) * torch.ones_like(x)
    return n.contiguous(), u.contiguous()


def _ensemble(c, seed):
    """Sizes and physics of a parameter sweep (the ranges of the batch workload)."""
    g = _gen(1000003 + c["count"])       # the ensemble is fixed; the seed changes its states
    out = []
    for i in range(c["count"]):
        nx = 32 * int(g.integers(4, c["nx_max"] // 32 + 1))
        ny = 16 * int(g.integers(4, c["ny_max"] // 16 + 1))
        out.append({"nx": nx, "ny": ny, "walls": True, "uw": float(g.uniform(0.0, 0.1)), "a0": float(g.uniform(1e-4, 5e-4)),
                    "lam": float((32, 64)[int(g.integers(0, 2))]), "tr": float(g.uniform(0.92, 0.96)), "tau": 1.0,
                    "start": "noise", "seed": int(seed) * 1000 + i})
    return out


def _params(c, prec):
    return lbm.lb_params(c["nx"], c["ny"], int(c["walls"]), PREC[prec], A_VDW, B_VDW, c["tr"] * T_C, KAPPA, c["tau"], c["a0"],
                         c["lam"], -c["uw"], c["uw"], ST_N, ST_Q, 0.0, None)


def _solver(c, prec):
    return lbm.Solver(c["nx"], c["ny"], walls=c["walls"], precision=PREC[prec], a=A_VDW, b=B_VDW, T=c["tr"] * T_C,
                      kappa=KAPPA, tau=c["tau"], A0=c["a0"], lam=c["lam"], u_bot=-c["uw"], u_top=c["uw"], N=ST_N, Q=ST_Q)


def _weights(seed):
    """Seeded initial weights in the order of include/fno.h (float32)."""
    g = _gen(seed)
    parts = [g.standard_normal((WIDTH, 5)) / math.sqrt(5.0), 0.1 * g.standard_normal(WIDTH)]
    for _ in range(LAYERS):
        parts += [g.standard_normal((WIDTH, WIDTH)) / math.sqrt(WIDTH), 0.1 * g.standard_normal(WIDTH),
                  g.uniform(0, 1, (MY, MX, WIDTH, WIDTH)) / WIDTH ** 2, g.uniform(0, 1, (MY, MX, WIDTH, WIDTH)) / WIDTH ** 2]
    parts += [g.standard_normal((HIDDEN, WIDTH)) / math.sqrt(WIDTH), 0.1 * g.standard_normal(HIDDEN),
              g.standard_normal((OUT, HIDDEN)) / math.sqrt(HIDDEN), 0.1 * g.standard_normal(OUT)]
    return np.concatenate([p.ravel() for p in parts]).astype(np.float32)


def _draws(n, seed):
    """Problem parameters (U_w, A0, lambda, T_r) of the warm-start range."""
    g = _gen(seed + 77)
    return np.stack([g.uniform(0.0, 0.035, n), g.uniform(3e-4, 1e-3, n), np.where(g.integers(0, 2, n) == 0, 32.0, 64.0),
                     g.uniform(0.925, 0.96, n)], axis=1).astype(np.float32)


def _targets(c, seed):
    """Settled striped fields as the network sees them (scaled n, u_x, u_y)."""
    dev = _dev()
    tg = torch.Generator(device=dev)
    tg.manual_seed(int(seed) + 5)
    y = torch.linspace(-1.0, 1.0, c["ny"], device=dev)[None, :, None]
    x = torch.linspace(0.0, 2.0 * math.pi, c["nx"] + 1, device=dev)[None, None, :-1]
    ph, h = torch.rand((2, c["batch"], 1, 1), device=dev, generator=tg)
    n = torch.tanh((y - 0.8 * (h - 0.5) + 0.05 * torch.cos(4.0 * x + 6.0 * ph)) * 12.0)
    ux = (0.6 * y + 0.05 * torch.sin(4.0 * x + 6.0 * ph)) * torch.ones_like(n)
    uy = 0.05 * torch.cos(4.0 * x + 6.0 * ph) * (1.0 - y * y)
    return torch.stack([n, ux, uy], dim=1).float().contiguous()


def prepare(case, seed):
    c, k = case, case["kind"]
    if k in ("flow", "monitor"):
        s = _solver(c, c["prec"])
        if c["tune"]:
            s.init_noise(1, 1.0, NOISE)
            s.autotune(20)
        st = {"case": c, "seed": int(seed), "solver": s}
        f64 = c["prec"] == "fp64"
        if c["start"] == "stripes":
            st["n0"], st["u0"] = _stripes(c, seed)
        if k == "flow":
            st["fields"] = torch.empty((3, c["ny"], c["nx"]), dtype=torch.float64 if f64 else torch.float32, device="cuda")
            if f64:
                st["sums"] = torch.zeros(5, dtype=torch.float64).pin_memory()
        else:
            n0 = st.pop("n0").cpu() if "n0" in st else torch.from_numpy(_noise(c, seed))
            st["host_n0"] = n0.pin_memory()
            st["host_fields"] = torch.zeros((3, c["ny"], c["nx"]), dtype=torch.float32).pin_memory()
            st["ring"] = torch.zeros((c["steps"], 6), dtype=torch.float64).pin_memory()
            try:
                s.monitor(st["ring"])
            except lbm.LBError:          # sizes that the monitored kernel does not take
                st["ring"] = None
        return st
    if k == "batch":
        cs = _ensemble(c, seed)
        b = lbm.Batch([_params(m, c["prec"]) for m in cs])
        return {"case": c, "members": cs, "batch": b,
                "fields": [torch.empty((3, m["ny"], m["nx"]), dtype=torch.float32, device="cuda") for m in cs]}
    net = fno_mod.Fno(width=WIDTH, hidden=HIDDEN, layers=LAYERS, modes_x=MX, modes_y=MY, outputs=OUT, batch_max=c["batch"],
                      nx_max=c["nx"], ny_max=c["ny"], gemm_bf16=True)
    net.set_params(_weights(seed))
    prm = torch.from_numpy(_draws(c["batch"], seed)).cuda()
    out = torch.empty((c["batch"], OUT, c["ny"], c["nx"]), dtype=torch.float32, device="cuda")
    st = {"case": c, "net": net, "prm": prm, "out": out}
    if k == "train":
        st["target"] = _targets(c, seed)
        st["grads"], st["weights"] = (torch.zeros(net.n_params, dtype=torch.float32).pin_memory() for _ in range(2))
    else:
        st["start"] = torch.empty((c["batch"], 3, c["ny"], c["nx"]), dtype=torch.float64, device="cuda")
        st["fields"] = torch.empty((c["batch"], 3, c["ny"], c["nx"]), dtype=torch.float32, device="cuda")
        p = _draws(c["batch"], seed).astype(np.float64)
        st["solvers"] = [_solver({"nx": c["nx"], "ny": c["ny"], "walls": True, "uw": p[i, 0], "a0": p[i, 1], "lam": p[i, 2],
                                  "tr": p[i, 3], "tau": 1.0}, "fp32") for i in range(c["batch"])]
    return st


# -------------------------------------------------------------------- runs

def run(state):
    c, k = state["case"], state["case"]["kind"]
    if k == "flow":
        s, m = state["solver"], state["fields"]
        if c["start"] == "stripes":
            s.init_fields(state["n0"], state["u0"])
        else:
            s.init_noise(state["seed"], 1.0, NOISE)
        s.step(c["steps"])
        lbm.lb_moments(s.h, m[0], m[1], m[2], lbm.LB_DTYPE_F64 if c["prec"] == "fp64" else lbm.LB_DTYPE_F32, 1)
        if c["prec"] != "fp64":
            return {"fields": m}
        lbm.lb_reduce_async(s.h, state["sums"])
        return {"fields": m, "sums": state["sums"]}
    if k == "monitor":
        s, m = state["solver"], state["host_fields"]
        s.init_fields(state["host_n0"])
        s.step(c["steps"])
        lbm.lb_moments(s.h, m[0], m[1], m[2], lbm.LB_DTYPE_F32, 0)
        return {"fields": m} if state["ring"] is None else {"fields": m, "records": state["ring"].float()}
    if k == "batch":
        b = state["batch"]
        for v, m in zip(b, state["members"]):
            v.init_noise(m["seed"], 1.0, NOISE)
        b.step(c["steps"])
        for v, m in zip(b, state["fields"]):
            lbm.lb_moments(v.h, m[0], m[1], m[2], lbm.LB_DTYPE_F32, 1)
        # one flat array of every lattice's fields
        return {"fields": torch.cat([m.reshape(-1) for m in state["fields"]])}
    net = state["net"]
    net.forward(state["prm"], c["nx"], c["ny"], state["out"])
    if k == "train":
        net.backward(state["target"], want_loss=False)
        net.adam(LR)
        fno_mod.fno_get_grads(net.h, state["grads"].numpy())
        fno_mod.fno_get_params(net.h, state["weights"].numpy())
        return {"out": state["out"], "grads": state["grads"], "weights": state["weights"]}
    net.fields(state["out"], c["nx"], c["ny"], SCALES, 1.0, state["start"])
    for i, s in enumerate(state["solvers"]):
        f, m = state["start"][i], state["fields"][i]
        s.init_fields(f[0], f[1], f[2])
        lbm.lb_moments(s.h, m[0], m[1], m[2], lbm.LB_DTYPE_F32, 1)
    return {"out": state["out"], "fields": state["fields"]}


# -------------------------------------------------------------------- work

STEP_FLOPS = 250.0                       # one site update: sums, stencils, force, equilibrium, forcing, collision


def _flow_work(c, prec, host=False):
    sites, pop = c["nx"] * c["ny"], SITE_BYTES[prec]
    out = 3 * (8 if prec == "fp64" else 4)
    start = pop + (8 if host or c.get("start") == "stripes" else 0) + (8 if c.get("start") == "stripes" else 0)
    # initial state written, every step one read and one write of the populations, moments read and written
    b = sites * (start + 2.0 * pop * c["steps"] + pop + out) + (sites * pop if prec == "fp64" else 0)
    return {"bytes": float(b), "flops": float(sites * STEP_FLOPS * c["steps"])}


def _net_flops(c):
    s = c["batch"] * c["nx"] * c["ny"]
    lines = c["batch"] * WIDTH * c["ny"]
    layer = 2 * lines * c["nx"] * 2 * MX * 2 + 2 * s * WIDTH * WIDTH + 16 * lines * MX * MY + 8 * c["batch"] * MX * MY * WIDTH ** 2
    return float(LAYERS * layer + 2 * s * WIDTH * 5 + 2 * s * HIDDEN * WIDTH + 2 * s * HIDDEN * OUT)


def _n_params():
    return WIDTH * 6 + LAYERS * (WIDTH * WIDTH + WIDTH + 2 * MX * MY * WIDTH * WIDTH) + HIDDEN * WIDTH + HIDDEN + OUT * HIDDEN + OUT


def work(case):
    c, k = case, case["kind"]
    if k in ("flow", "monitor"):
        return _flow_work(c, c["prec"], k == "monitor")
    if k == "batch":
        w = [_flow_work({**m, "steps": c["steps"]}, c["prec"]) for m in _ensemble(c, 0)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    s = c["batch"] * c["nx"] * c["ny"]
    if k == "train":                     # weights and moments read and written, gradients written, output and target
        return {"bytes": float(4 * _n_params() * 9 + 2 * 4 * OUT * s), "flops": 3.0 * _net_flops(c)}
    return {"bytes": float(4 * _n_params() + s * (4 * OUT + 2 * 24 + 2 * 36 + 12)), "flops": _net_flops(c) + 100.0 * s}


# ------------------------------------------------- the same in 64 bits (torch)

def _noise(c, seed):
    """The noisy uniform start of lb_init mode 0: SplitMix64 output k of the seed."""
    k = np.arange(c["nx"] * c["ny"], dtype=np.uint64)
    with np.errstate(over="ignore"):
        z = np.uint64(int(seed)) + (k + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    u = (z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
    return (1.0 + NOISE * (2.0 * u - 1.0)).reshape(c["ny"], c["nx"])


CX, CY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
W9 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
T0 = 1.0 / 3.0


def _feq(n, u, v, T):
    out, uu = [], u * u + v * v
    for i in range(9):
        cu = CX[i] * u + CY[i] * v
        cc = CX[i] ** 2 + CY[i] ** 2
        out.append(W9[i] * n * (1.0 + cu / T0 + (cu * cu - T0 * uu) / (2 * T0 * T0) + (T - T0) * (cc - 2 * T0) / (2 * T0 * T0)))
    return out


class _Ref:
    """The scheme in torch FP64 on whole fields."""

    def __init__(self, c, n0, u0=None, v0=None):
        self.c, self.T, self.walls = c, c["tr"] * T_C, bool(c["walls"])
        z = torch.zeros_like(n0)
        self.f = _feq(n0, z if u0 is None else u0, z if v0 is None else v0, self.T)
        x = torch.arange(c["nx"], dtype=torch.float64, device=n0.device)
        self.fx = (c["a0"] * torch.sin(2.0 * math.pi * x / c["lam"]))[None, :]

    def at(self, a, dx, dy, odd=False):
        """a at (x + dx, y + dy): periodic, or mirrored about the wall rows."""
        if dy:
            if self.walls:
                g = a[1:2] if dy < 0 else a[-2:-1]
                g = -g if odd else g
                a = torch.cat([g, a[:-1]]) if dy < 0 else torch.cat([a[1:], g])
            else:
                a = torch.roll(a, -dy, 0)
        return torch.roll(a, -dx, 1) if dx else a

    def grad(self, a, odd=False):
        m = (1.0 - 2.0 * ST_N) / 4.0
        p = [self.at(a, CX[i], CY[i], odd) for i in range(9)]
        return (ST_N * (p[1] - p[3]) + m * ((p[5] - p[6]) + (p[8] - p[7])),
                ST_N * (p[2] - p[4]) + m * ((p[5] - p[8]) + (p[6] - p[7])))

    def lap(self, a):
        r = (1.0 - ST_Q) / 2.0
        p = [self.at(a, CX[i], CY[i]) for i in range(9)]
        return ST_Q * (p[1] + p[2] + p[3] + p[4]) + r * (p[5] + p[6] + p[7] + p[8]) - 4.0 * (ST_Q + r) * a

    def moments(self):
        f = self.f
        g = [torch.roll(f[i], (CY[i], CX[i]), (0, 1)) for i in range(9)]
        n = sum(g)
        if self.walls:
            n[0] = (f[0][0] + f[4][0] + f[7][0] + f[8][0]) + (g[1][0] + g[3][0] + g[4][0] + g[7][0] + g[8][0])
            n[-1] = (f[0][-1] + f[2][-1] + f[6][-1] + f[5][-1]) + (g[1][-1] + g[3][-1] + g[2][-1] + g[6][-1] + g[5][-1])
        P = n * self.T - (n * self.T / (1.0 - B_VDW * n) - A_VDW * n * n)
        (px, py), (lx, ly) = self.grad(P), self.grad(self.lap(n))
        Fx, Fy = px + KAPPA * n * lx + self.fx, py + KAPPA * n * ly
        if self.walls:
            for r, s in ((0, 1.0), (-1, -1.0)):      # bottom, then the y-mirror on top
                U = -self.c["uw"] if r == 0 else self.c["uw"]
                i4, i7, i8, i5, i6, i2 = (4, 7, 8, 5, 6, 2) if r == 0 else (2, 6, 5, 8, 7, 4)
                d = 0.5 * (g[1][r] - g[3][r])
                fy = s * Fy[r]
                g[0][r] = n[r] - (g[1][r] + g[3][r]) - 2.0 * (g[i4][r] + g[i7][r] + g[i8][r]) + 0.5 * fy
                g[i5][r] = g[i7][r] - d - 0.25 * (Fx[r] + fy) + 0.5 * n[r] * U
                g[i6][r] = g[i8][r] + d + 0.25 * (Fx[r] - fy) - 0.5 * n[r] * U
                g[i2][r] = g[i4][r]
        Jx = g[1] - g[3] + g[5] - g[6] - g[7] + g[8] + 0.5 * Fx
        Jy = g[2] - g[4] + g[5] + g[6] - g[7] - g[8] + 0.5 * Fy
        return n, Jx, Jy, Fx, Fy, g

    def step(self):
        n, Jx, Jy, Fx, Fy, g = self.moments()
        u, v, tau = Jx / n, Jy / n, self.c["tau"]
        (nx_, ny_), div = self.grad(n), self.grad(Jx)[0] + self.grad(Jy, odd=True)[1]
        fe, q, th = _feq(n, u, v, self.T), 1.0 - 0.5 / tau, T0 - self.T
        cxx = q * (2.0 * u * Fx + th * (2.0 * u * nx_ + div))
        cyy = q * (2.0 * v * Fy + th * (2.0 * v * ny_ + div))
        cxy = q * (u * Fy + v * Fx + th * (u * ny_ + v * nx_))
        for i in range(9):
            cc = cxx * CX[i] ** 2 + 2.0 * cxy * CX[i] * CY[i] + cyy * CY[i] ** 2
            Fi = W9[i] * (q * (CX[i] * Fx + CY[i] * Fy) / T0 + (cc - T0 * (cxx + cyy)) / (2 * T0 * T0))
            g[i] = g[i] - (g[i] - fe[i]) / tau + Fi
        self.f = g

    def run(self, steps):
        for _ in range(steps):
            self.step()
        n, Jx, Jy = self.moments()[:3]
        return torch.stack([n, Jx / n, Jy / n])


def _ref_fields(c, seed):
    if c["start"] == "stripes":
        n0, u0 = _stripes(c, seed)
        return _Ref(c, n0, None if c["kind"] == "monitor" else u0)
    return _Ref(c, torch.from_numpy(_noise(c, seed)).to(_dev()))


def _unpack(flat):
    shapes = [(WIDTH, 5), (WIDTH,)] + [(WIDTH, WIDTH), (WIDTH,), (MY, MX, WIDTH, WIDTH), (MY, MX, WIDTH, WIDTH)] * LAYERS + \
        [(HIDDEN, WIDTH), (HIDDEN,), (OUT, HIDDEN), (OUT,)]
    out, at = [], 0
    for s in shapes:
        n = int(np.prod(s))
        out.append(flat[at:at + n].reshape(s))
        at += n
    return out


def _net64(flat, prm, nx, ny):
    """The network of include/fno.h in FP64."""
    p, dev = _unpack(flat), flat.device
    B = prm.shape[0]
    x = torch.arange(nx, dtype=torch.float64, device=dev)[None, None, :]
    y = (2.0 * torch.arange(ny, dtype=torch.float64, device=dev) / (ny - 1) - 1.0)[None, :, None]
    uw, a0, lam, tr = (prm[:, j, None, None].double() for j in range(4))
    one = torch.ones((B, ny, nx), dtype=torch.float64, device=dev)
    v = torch.stack([a0 / 1e-3 * torch.sin(2.0 * math.pi * x / lam) * one, a0 / 1e-3 * torch.cos(2.0 * math.pi * x / lam) * one,
                     uw / 0.05 * y * one, (tr - 0.94) / 0.02 * one, y * one], dim=1)
    lin = lambda w, a: torch.einsum("oc,bcyx->boyx", w, a)  # noqa: E731
    gelu = lambda a: a * 0.5 * (1.0 + torch.erf(a / math.sqrt(2.0)))  # noqa: E731
    v = lin(p[0], v) + p[1][None, :, None, None]
    kx = torch.arange(MX, dtype=torch.float64, device=dev)
    ky = torch.cat([torch.arange(MY // 2), torch.arange(-(MY // 2), 0)]).to(dev, torch.float64)
    ex = torch.polar(torch.ones(MX, nx, dtype=torch.float64, device=dev), 2.0 * math.pi * kx[:, None] * x[0] / nx)
    ey = torch.polar(torch.ones(MY, ny, dtype=torch.float64, device=dev),
                     2.0 * math.pi * ky[:, None] * torch.arange(ny, dtype=torch.float64, device=dev)[None, :] / ny)
    ck = torch.where(kx == 0, 1.0, 2.0)
    for l in range(LAYERS):
        W, w, Rr, Ri = p[2 + 4 * l:6 + 4 * l]
        vh = torch.einsum("bcyk,my->bcmk", torch.einsum("bcyx,kx->bcyk", v + 0j, ex.conj()), ey.conj())
        s = torch.einsum("bcmk,mkco->bomk", vh, torch.complex(Rr, Ri))
        s = torch.einsum("bomk,my->boyk", s, ey) * ck
        z = torch.einsum("boyk,kx->boyx", s, ex).real / (nx * ny)
        z = lin(W, v) + w[None, :, None, None] + z
        v = gelu(z) if l < LAYERS - 1 else z
    h = gelu(lin(p[-4], v) + p[-3][None, :, None, None])
    return lin(p[-2], h) + p[-1][None, :, None, None]


def exact(case, seed):
    c, k = case, case["kind"]
    with torch.no_grad():
        if k in ("flow", "monitor"):
            r = _ref_fields(c, seed)
            m = r.run(c["steps"])
            if k == "monitor":
                return {"fields": m, "records": None}
            if c["prec"] != "fp64":
                return {"fields": m}
            s = [sum(f.sum() for f in r.f), sum(CX[i] * r.f[i].sum() for i in range(9)),
                 sum(CY[i] * r.f[i].sum() for i in range(9))]
            return {"fields": m, "sums": torch.stack([t.double() for t in s] + [torch.zeros_like(s[0])] * 2)}
        if k == "batch":
            if c["count"] * c["steps"] > 3200:
                return None
            return {"fields": torch.cat([_Ref(m, torch.from_numpy(_noise(m, m["seed"])).to(_dev())).run(c["steps"]).reshape(-1)
                                         for m in _ensemble(c, seed)])}
    flat = torch.from_numpy(_weights(seed)).to(_dev()).double()
    prm = torch.from_numpy(_draws(c["batch"], seed)).to(_dev())
    if k == "train":
        flat.requires_grad_(True)
        out, target, grads = [], _targets(c, seed).double(), torch.zeros_like(flat)
        for b in range(c["batch"]):      # field by field: the FP64 graph of one field at a time
            o = _net64(flat, prm[b:b + 1], c["nx"], c["ny"])
            grads += torch.autograd.grad(((o - target[b:b + 1]) ** 2).sum() / target.numel(), flat)[0]
            out.append(o.detach())
        return {"out": torch.cat(out), "grads": grads, "weights": None}
    with torch.no_grad():
        out = torch.cat([_net64(flat, prm[b:b + 1], c["nx"], c["ny"]) for b in range(c["batch"])])
        fields = []
        for b in range(c["batch"]):
            n = 1.0 + SCALES[0] * out[b, 0]
            uw, a0, lam, tr = (float(v) for v in _draws(c["batch"], seed)[b].astype(np.float64))
            q = {"nx": c["nx"], "ny": c["ny"], "walls": True, "uw": uw, "a0": a0, "lam": lam, "tr": tr, "tau": 1.0}
            r = _Ref(q, n + (1.0 - n.mean()), SCALES[1] * out[b, 1], SCALES[2] * out[b, 2])
            fields.append(r.run(0))
        return {"out": out, "fields": torch.stack(fields)}
