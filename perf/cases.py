"""Performance cases: the work this framework is used for, through its public entry points.

Cells (`Sim`) stepped in blocks with their fields and Nusselt number read after each block, ensembles (`Batch`)
stepped and sampled as the training-data and evaluation loops do, the diagnostics of a large state, and the
learned warm start's training iteration, single layers and prediction.  Every state starts from a developed-looking
flow: convection rolls of random strength plus noise, handed over as T and u fields (`tlbm_init_fields`).
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2211_03160_gb300 import surrogate, tlbm

MA = 0.1
U_FF = MA / math.sqrt(3.0)  # free-fall velocity in lattice units
BYTES = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}
# operations of one lattice update in its two-relaxation-time form (sums, velocity, equilibria, pair updates)
FLOPS_LU = {2: 150, 3: 330}


def _cell(name, shape, precision, Ra, steps, nu=False, inplace=False, walls="rb", periodic=0, Pr=0.71):
    shape = tuple(shape) + (1,) * (3 - len(shape))
    return {"name": name, "kind": "cell", "dim": 3 if shape[2] > 1 else 2, "nx": shape[0], "ny": shape[1],
            "nz": shape[2], "precision": precision, "Ra": Ra, "Pr": Pr, "steps": steps, "nu": nu,
            "inplace": inplace, "walls": walls, "periodic": periodic}


def _ensemble(name, count, sizes, precision, steps, tune, log_ra_lo=5.0, log_ra_hi=8.0):
    return {"name": name, "kind": "ensemble", "count": count, "sizes": sizes, "precision": precision, "steps": steps,
            "tune": tune, "log_ra_lo": log_ra_lo, "log_ra_hi": log_ra_hi, "draw_seed": 4}


def listed():
    return [
        # the validation cell: the oracle-compared FP64 run, launch- and latency-bound
        _cell("cell2d_129_fp64", (129, 129), "fp64", 1e5, 1000, nu=True),
        # a small chaotic cell sampled 16 times per free-fall time (4452 steps), as the precision study does
        _cell("cell2d_257_fp32", (257, 257), "fp32", 1e7, 278, nu=True),
        # the headline cell in its two benchmark storages: a block of steps, then the fields
        _cell("cell2d_8193_fp32", (8193, 8193), "fp32", 1e8, 32),
        _cell("cell2d_8193_fp16", (8193, 8193), "fp16", 1e8, 32),
        # the paper's own precision on a large cell
        _cell("cell2d_4097_fp64", (4097, 4097), "fp64", 1e8, 16),
        # the 3D cube in its two benchmark storages, and in the paper's precision
        _cell("cube_385_fp32", (385, 385, 385), "fp32", 1e7, 32),
        _cell("cube_385_fp16", (385, 385, 385), "fp16", 1e7, 32),
        _cell("cube_193_fp64", (193, 193, 193), "fp64", 1e6, 16),
        # the 64-cell ensemble as the training-data loop uses it (FP32, launch shape left to the library), and as the
        # benchmark does (FP16, tuned once); fields and Nusselt numbers of every cell after each block
        _ensemble("ensemble64_fp32", 64, "129,257,513,1025", "fp32", 32, False),
        _ensemble("ensemble64_fp16", 64, "129,257,513,1025", "fp16", 32, True),
        # monitoring a large run: fields, Nusselt number, kinetic energy and mass of the current state
        {"name": "monitor2d_8193_fp32", "kind": "monitor", "dim": 2, "nx": 8193, "ny": 8193, "nz": 1,
         "precision": "fp32", "Ra": 1e8, "Pr": 0.71, "inplace": False, "walls": "rb", "periodic": 0},
        # one full-batch training iteration of the warm-start network on its 48 samples
        {"name": "train_48x65", "kind": "train", "batch": 48, "n": 65},
    ]


def _odd(rng, lo, hi):
    """Log-uniform in [lo, hi], odd more often than not."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return v | 1 if rng.random() < 0.75 else v


def draw(rng):
    kind = rng.choices(["cell2d", "cell3d", "ensemble", "monitor", "train", "layer", "start"],
                       [5, 4, 3, 1, 1, 1, 1])[0]
    if kind in ("cell2d", "cell3d", "monitor"):
        dim = 3 if kind == "cell3d" or (kind == "monitor" and rng.random() < 0.4) else 2
        precision = rng.choices(["fp64", "fp32", "fp16", "bf16"], [3, 4, 3, 1])[0]
        top = {2: 2000 if precision == "fp64" else 8193, 3: 161 if precision == "fp64" else 385}[dim]
        n = _odd(rng, 65 if dim == 2 else 33, top)
        shape = [n] + [min(top, max(17, int(n * rng.uniform(0.6, 1.0)))) | 1 for _ in range(dim - 1)]
        rng.shuffle(shape)
        shape = tuple(shape) + (1,) * (3 - dim)
        nodes = shape[0] * shape[1] * shape[2]
        # the least viscous cell kept: nu about 0.004, stable at every size
        h = shape[dim - 1]
        Ra = min(1e8, 0.71 * (U_FF * h / 0.004) ** 2) * rng.uniform(0.1, 1.0)
        walls = "side" if rng.random() < 0.2 else "rb"
        periodic = rng.choice([1, 1, 3 if dim == 3 and walls == "rb" else 1]) if walls == "rb" and rng.random() < 0.2 else 0
        inplace = rng.random() < 0.2
        if kind == "monitor":
            return {"kind": "monitor", "dim": dim, "nx": shape[0], "ny": shape[1], "nz": shape[2],
                    "precision": precision, "Ra": Ra, "Pr": 0.71, "inplace": inplace, "walls": walls,
                    "periodic": periodic}
        budget = 6e7 if precision == "fp64" else 1e9  # lattice updates of a pass
        if dim == 3:
            budget /= 2
        most = 64 if precision in ("fp16", "bf16") else 512
        steps = max(3, min(most, int(budget / nodes * rng.uniform(0.4, 1.0))))
        c = _cell("", shape, precision, Ra, steps, nu=rng.random() < 0.5, inplace=inplace, walls=walls,
                  periodic=periodic, Pr=rng.choice([0.71, 0.71, 7.0]))
        c.pop("name")
        return c
    if kind == "ensemble":
        sizes = rng.choice(["129,257,513,1025", "65", "513", "129,257", "97,161,321,641", "257,513,1025"])
        c = _ensemble("", rng.randint(6, 64), sizes, rng.choice(["fp32", "fp32", "fp16", "bf16"]),
                      rng.choice([16, 24, 32, 37]), rng.random() < 0.4)
        c.pop("name")
        c["draw_seed"] = rng.randint(5, 1000)
        return c
    if kind == "train":
        return {"kind": "train", "batch": rng.randint(4, 64), "n": rng.choice([33, 65, 65, 97])}
    if kind == "layer":
        cin, cout = rng.choice([(5, 32), (32, 32), (32, 32), (32, 3), (17, 24)])
        return {"kind": "layer", "batch": rng.randint(1, 48), "cin": cin, "cout": cout, "h": _odd(rng, 17, 129),
                "w": _odd(rng, 17, 260)}
    return {"kind": "start", "fine": rng.choice([129, 257, 513, 1025]), "precision": rng.choice(["fp32", "fp16"]),
            "Ra": 10.0 ** rng.uniform(5.0, 6.0), "Pr": rng.choice([0.71, 7.0])}


# ------------------------------------------------------------------ inputs


def _rolls(dim, shape, seed, side=False):
    """T, ux, uy[, uz] (FP32, on the GPU): the conductive profile, rolls of random strength and phase, noise."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    r = np.random.default_rng(int(seed))
    nx, ny, nz = shape
    ax = [((torch.arange(n, device="cuda", dtype=torch.float32) + 0.5) / n) for n in (nx, ny, nz)]
    if dim == 2:
        x, y = ax[0][None, :], ax[1][:, None]
        c = x if side else y
    else:
        x, y, z = ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]
        c = x if side else z
    v = y if dim == 2 else z  # the vertical coordinate
    full = (ny, nx) if dim == 2 else (nz, ny, nx)
    T = (0.5 - c).expand(full).clone()
    u = [torch.zeros(full, device="cuda") for _ in range(dim)]
    for j in range(2):
        k, m = int(r.integers(1, 4)), int(r.integers(1, 3))
        a, b = r.uniform(0.2, 0.5) * U_FF, r.uniform(0.05, 0.15)
        hor, wave = (0, x) if dim == 2 or j == 0 else (1, y)  # in 3D one set of rolls along each horizontal axis
        s, t = torch.sin(math.pi * k * wave), torch.cos(math.pi * k * wave)
        p, q = torch.sin(math.pi * m * v), torch.cos(math.pi * m * v)
        u[hor] += a * s * q
        u[-1] -= a * t * p
        T += b * t * p
    T += 2e-3 * (torch.rand(full, generator=g, device="cuda") - 0.5)
    for w in u:
        w += 2e-4 * U_FF * (torch.rand(full, generator=g, device="cuda") - 0.5)
    return T, u


def _sim(case, seed):
    dim = case["dim"]
    sim = tlbm.Sim(case["nx"], case["ny"], case["nz"],
                   lattice=tlbm.TLBM_D2Q9_D2Q5 if dim == 2 else tlbm.TLBM_D3Q19_D3Q7, Ra=case["Ra"], Pr=case["Pr"],
                   Ma=MA, precision=tlbm.PRECISIONS[case["precision"]],
                   walls=tlbm.TLBM_SIDE_HEATED if case["walls"] == "side" else tlbm.TLBM_RB,
                   periodic_mask=case["periodic"],
                   streaming=tlbm.TLBM_STREAM_INPLACE if case["inplace"] else tlbm.TLBM_STREAM_PULL)
    T, u = _rolls(dim, (case["nx"], case["ny"], case["nz"]), seed, case["walls"] == "side")
    tlbm.tlbm_init_fields(sim.h, T, *u)
    return sim


def _members(case):
    """(n, Ra, Pr, seed) of an ensemble's cells: sizes, Ra (log-uniform) and Pr drawn as in the ensemble benchmark."""
    r = np.random.default_rng(case["draw_seed"])
    sizes = [int(s) for s in case["sizes"].split(",")]
    return [(int(r.choice(sizes)), float(10.0 ** r.uniform(case["log_ra_lo"], case["log_ra_hi"])),
             float(r.choice((0.71, 7.0))), 100 + i) for i in range(case["count"])]


def _net(seed):
    """A network in mid-training: weights, biases and optimiser moments away from zero."""
    net = surrogate.ConvNet(seed=int(seed) % (1 << 31))
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    rnd = lambda t, s: s * torch.randn(t.shape, generator=g, device="cuda")  # noqa: E731
    for k in range(len(net.shapes)):
        net.b[k].copy_(rnd(net.b[k], 0.05))
        for m, v in ((net.mw[k], net.vw[k]), (net.mb[k], net.vb[k])):
            m.copy_(rnd(m, 1e-3))
            v.copy_(1e-5 + rnd(v, 2e-3).square())
    net.t = 100
    return net


def _train_data(case, seed):
    """BF16 inputs and FP32 targets of a batch: smooth fields and the two parameter channels."""
    B, n = case["batch"], case["n"]
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 7)
    low = torch.rand((B, 6, 5, 5), generator=g, device="cuda") - 0.5
    fields = F.interpolate(low, size=(n, n), mode="bilinear", align_corners=True)
    par = (torch.rand((B, 2, 1, 1), generator=g, device="cuda") * 2 - 1).expand(B, 2, n, n)
    x = torch.cat([fields[:, :3], par], 1).to(torch.bfloat16).contiguous()
    return x, fields[:, 3:].contiguous()


def _layer_data(case, seed):
    B, ci, co, h, w = (case[k] for k in ("batch", "cin", "cout", "h", "w"))
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    x = torch.randn((B, ci, h, w), generator=g, device="cuda").relu().to(torch.bfloat16)
    wt = torch.randn((co, ci, 3, 3), generator=g, device="cuda") * math.sqrt(2.0 / (9 * ci))
    b = 0.05 * torch.randn(co, generator=g, device="cuda")
    dy = 1e-3 * torch.randn((B, co, h, w), generator=g, device="cuda")
    return x, wt, b, dy


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("cell", "monitor"):
        return {"case": case, "sim": _sim(case, seed)}
    if kind == "ensemble":
        mem = _members(case)
        b = tlbm.Batch([(n, n, 1, Ra, Pr, MA, s) for n, Ra, Pr, s in mem],
                       precision=tlbm.PRECISIONS[case["precision"]])
        b.init(1e-3)
        for k, (n, _, _, s) in enumerate(mem):
            T, u = _rolls(2, (n, n, 1), int(seed) * 1000 + s)
            tlbm.tlbm_init_fields(b.instance(k), T, *u)
        if case["tune"]:
            b.autotune()
        nodes = sum(n * n for n, *_ in mem)
        out = {k: torch.empty(nodes, dtype=torch.float32, device="cuda") for k in ("T", "ux", "uy")}
        at = np.concatenate([[0], np.cumsum([n * n for n, *_ in mem])]).tolist()
        views = [tuple(out[k][at[i]:at[i + 1]] for k in ("ux", "uy", "T")) for i in range(len(mem))]
        return {"case": case, "batch": b, "out": out, "views": views}
    if kind == "train":
        x16, tgt = _train_data(case, seed)
        return {"case": case, "net": _net(seed), "x16": x16, "tgt": tgt, "g32": torch.empty_like(tgt),
                "g16": torch.empty(tgt.shape, dtype=torch.bfloat16, device="cuda"),
                "loss": torch.zeros(1, dtype=torch.float64, device="cuda"),
                "part": torch.zeros(1024, dtype=torch.float64, device="cuda")}
    if kind == "layer":
        B, ci, co, h, w = (case[k] for k in ("batch", "cin", "cout", "h", "w"))
        x, wt, b, dy = _layer_data(case, seed)
        a = torch.empty(tlbm.tlbm_conv3x3_weight_elems(ci), dtype=torch.bfloat16, device="cuda")
        tlbm.tlbm_conv3x3_pack_weights(wt, co, ci, a, torch.cuda.current_stream())
        e = lambda *s, t=torch.float32: torch.empty(s, dtype=t, device="cuda")  # noqa: E731
        return {"case": case, "x": x, "a": a, "b": b, "w16": wt.to(torch.bfloat16), "dy": dy,
                "dy16": dy.to(torch.bfloat16), "y": e(B, co, h, w), "act": e(B, co, h, w, t=torch.bfloat16),
                "dx": e(B, ci, h, w), "dw": e(co, ci, 3, 3), "db": e(co), "at": e(32 * 288, t=torch.bfloat16),
                "ws": e(tlbm.tlbm_conv3x3_workspace_bytes(B, ci, co, h, w), t=torch.uint8)}
    n = case["fine"]
    sim = tlbm.Sim(n, n, Ra=case["Ra"], Pr=case["Pr"], Ma=MA, precision=tlbm.PRECISIONS[case["precision"]])
    sim.init(int(seed), 1e-3)
    return {"case": case, "sim": sim, "net": _net(seed), "x": surrogate.features(case["Ra"], case["Pr"], fine=n)}


# ------------------------------------------------------------------ one pass


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "cell":
        sim = state["sim"]
        sim.step(case["steps"])
        out = sim.macros(_dtype(case))
        if case["nu"]:
            out["nu"] = sim.nusselt()
        return out
    if kind == "monitor":
        sim = state["sim"]
        out = sim.macros(_dtype(case))
        out["nu"] = sim.nusselt()
        out["ekin"], out["mass"] = sim.energy()
        return out
    if kind == "ensemble":
        b = state["batch"]
        b.step(case["steps"])
        for k, (ux, uy, T) in enumerate(state["views"]):
            tlbm.tlbm_batch_macros(b.b, k, None, ux, uy, None, T, tlbm.TLBM_OUT_F32)
        return dict(state["out"], nu=torch.tensor(b.nusselt(allow_diverged=True)))
    s = torch.cuda.current_stream()
    if kind == "train":
        net, B, n = state["net"], case["batch"], case["n"]
        y = net.forward(state["x16"], B, n, n)
        tlbm.tlbm_mse_loss(y, state["tgt"], y.numel(), state["g32"], state["g16"], state["loss"], state["part"], s)
        net.backward(state["g32"], state["g16"], B, n, n)
        net.adam(2e-3)
        return {"y": y, "loss": state["loss"], "gw": net.gw, "gb": net.gb, "w": net.w, "b": net.b}
    if kind == "layer":
        d = (case["batch"], case["cin"], case["cout"], case["h"], case["w"])
        tlbm.tlbm_conv3x3_forward(state["x"], state["a"], state["b"], state["y"], state["act"], *d, 1, s)
        tlbm.tlbm_conv3x3_backward_weight(state["x"], state["dy16"], state["dy"], state["dw"], state["db"], *d,
                                          state["ws"], s)
        tlbm.tlbm_conv3x3_backward_data(state["dy16"], state["w16"], state["dx"], *d, state["at"], s)
        return {k: state[k] for k in ("y", "act", "dx", "dw", "db")}
    sim = state["sim"]
    c = surrogate.predict(state["net"], case["Ra"], case["Pr"], case["fine"], state["x"])
    surrogate.warm_start(sim.h, c, U_FF, case["fine"])
    return {"coarse": c, "fields": sim.macros(torch.float32)}


# ------------------------------------------------------------------ work


def work(case):
    kind = case["kind"]
    if kind in ("cell", "monitor"):
        dim, nodes = case["dim"], case["nx"] * case["ny"] * case["nz"]
        q, fields = (14, 4) if dim == 2 else (26, 5)
        state, out = nodes * q * BYTES[case["precision"]], nodes * fields * (8 if case["precision"] == "fp64" else 4)
        if kind == "monitor":
            return {"bytes": state + out, "flops": nodes * 3 * q}
        return {"bytes": 2 * state + out, "flops": case["steps"] * nodes * FLOPS_LU[dim]}
    if kind == "ensemble":
        nodes = sum(n * n for n, *_ in _members(case))
        return {"bytes": 2 * nodes * 14 * BYTES[case["precision"]] + nodes * 12,
                "flops": case["steps"] * nodes * FLOPS_LU[2]}
    gemm = lambda B, ci, co, h, w: 2.0 * 9 * ci * co * B * h * w  # noqa: E731
    if kind == "train":
        B, n = case["batch"], case["n"]
        layers = [(5, 32), (32, 32), (32, 32), (32, 3)]
        flops = sum(gemm(B, ci, co, n, n) * (2 if k == 0 else 3) for k, (ci, co) in enumerate(layers))
        weights = sum(9 * ci * co + co for ci, co in layers)
        return {"bytes": B * n * n * (5 * 2 + 3 * 4 + 3 * 4) + weights * 4 * 7, "flops": flops}
    if kind == "layer":
        B, ci, co, h, w = (case[k] for k in ("batch", "cin", "cout", "h", "w"))
        px = B * h * w
        return {"bytes": px * (2 * ci + 2 * co + 4 * co + 4 * co + 2 * co + 4 * ci) + 9 * ci * co * 8,
                "flops": 3 * gemm(B, ci, co, h, w)}
    n, m = case["fine"], surrogate.COARSE
    return {"bytes": n * n * (14 * BYTES[case["precision"]] + 16) + 5 * m * m * 4,
            "flops": sum(gemm(1, ci, co, m, m) for ci, co in [(5, 32), (32, 32), (32, 32), (32, 3)])}


# ------------------------------------------------------------------ exact values in 64 bits

_E2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_E3 = [(0, 0, 0)] + [tuple(s if a == b else 0 for b in range(3)) for a in range(3) for s in (1, -1)] + \
      [tuple(s if c == a else (t if c == b else 0) for c in range(3))
       for a, b in ((0, 1), (0, 2), (1, 2)) for s in (1, -1) for t in (1, -1)]


class _Flow:
    """The thermal lattice Boltzmann step of one cell in plain FP64 torch: populations as deviations from the rest
    state, two relaxation times, Guo forcing, half-way wall rules."""

    def __init__(self, dim, shape, Ra, Pr, T, u, side, periodic):
        self.dim, self.side, self.periodic = dim, side, periodic
        H = shape[dim - 1]
        self.nu, self.alpha = U_FF * H * math.sqrt(Pr / Ra), U_FF * H / math.sqrt(Pr * Ra)
        self.gb = U_FF * U_FF / H
        self.omega = (4.0 - 2.0 / 3.0) / 10.0 if dim == 2 else (6.0 - 0.75) / 21.0
        self.sp = 1.0 / (3.0 * self.nu + 0.5)
        self.sm = 8.0 * (2.0 - self.sp) / (8.0 - self.sp)
        self.qm = 1.0 / (self.alpha / self.omega + 0.5)
        self.qp = 1.0 / (0.5 + 0.25 / (1.0 / self.qm - 0.5))
        self.L = shape[0] if side else H
        self.e = _E2 if dim == 2 else _E3
        w = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36} if dim == 2 else {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
        self.w = [w[sum(map(abs, e))] for e in self.e]
        self.opp = [self.e.index(tuple(-c for c in e)) for e in self.e]
        self.th = [i for i, e in enumerate(self.e) if sum(map(abs, e)) <= 1]  # the thermal set's velocities
        self.ax = [1, 0] if dim == 2 else [2, 1, 0]  # tensor dimension of x, y[, z]
        T, u = T.double(), [v.double() for v in u]
        uu = sum(v * v for v in u)
        self.f, self.g = [], []
        for e, wi in zip(self.e, self.w):
            eu = sum(c * v for c, v in zip(e, u) if c) + torch.zeros_like(uu)
            self.f.append(wi * (3.0 * eu + 4.5 * eu * eu - 1.5 * uu))
        wt = 0.5 * self.omega
        for i in self.th:
            eu = sum(c * v for c, v in zip(self.e[i], u) if c)
            self.g.append((1.0 - 2 * dim * wt) * T if i == 0 else wt * T + 0.5 * eu * T)

    def macros(self):
        drho = sum(self.f)
        T = sum(self.g)
        rho = 1.0 + drho
        Fz = rho * (self.gb * T)
        u = []
        for a in range(self.dim):
            j = sum(e[a] * f for e, f in zip(self.e, self.f) if e[a])
            u.append((j + 0.5 * Fz) / rho if a == self.dim - 1 else j / rho)
        return drho, rho, T, Fz, u

    def _shift(self, posts, k, thermal):
        """Population k at its pulling nodes: the neighbour's post-collision value, or the wall rule's."""
        e = self.e[k]
        o = self.opp[k]
        src = posts[k] if not thermal else posts[self.th.index(k)]
        back = posts[o] if not thermal else posts[self.th.index(o)]
        out = torch.roll(src, [c for c in e if c], [self.ax[a] for a in range(self.dim) if e[a]]) if any(e) else src
        for a in range(self.dim):
            if e[a] == 0 or (self.periodic >> a) & 1:
                continue
            d = self.ax[a]
            edge = 0 if e[a] == 1 else out.shape[d] - 1
            v = back.select(d, edge)
            if thermal and a == (0 if self.side else self.dim - 1):
                v = -v + self.omega * (0.5 if edge == 0 else -0.5)
            out.select(d, edge).copy_(v)
        return out

    def step(self):
        drho, rho, T, Fz, u = self.macros()
        uu, uF = sum(v * v for v in u), u[-1] * Fz
        sp, sm, hp, hm = self.sp, self.sm, 1.0 - 0.5 * self.sp, 1.0 - 0.5 * self.sm
        base = sp * (drho - 1.5 * rho * uu) - 3.0 * hp * uF
        f, g, post, tpost = self.f, self.g, [None] * len(self.e), [None] * len(self.th)
        for i, e in enumerate(self.e):
            o = self.opp[i]
            if i == 0:
                post[0] = (1.0 - sp) * f[0] + self.w[0] * base
            elif i < o:
                eu = sum(c * v for c, v in zip(e, u) if c)
                eF = e[-1] * Fz
                s = 0.5 * (f[i] + f[o])
                a = 0.5 * (f[i] - f[o])
                s = s - sp * s + self.w[i] * (base + eu * (4.5 * sp * rho * eu + 9.0 * hp * eF))
                a = a - sm * a + self.w[i] * (3.0 * sm * rho * eu + 3.0 * hm * eF)
                post[i], post[o] = s + a, s - a
        wt = 0.5 * self.omega
        for k, i in enumerate(self.th):
            e, o = self.e[i], self.opp[i]
            if i == 0:
                tpost[0] = g[0] - self.qp * (g[0] - (1.0 - 2 * self.dim * wt) * T)
            elif i < o:
                m = self.th.index(o)
                s, a = 0.5 * (g[k] + g[m]), 0.5 * (g[k] - g[m])
                eu = sum(c * v for c, v in zip(e, u) if c)
                s = s - self.qp * (s - wt * T)
                a = a - self.qm * (a - 0.5 * eu * T)
                tpost[k], tpost[m] = s + a, s - a
        self.f = [self._shift(post, i, False) for i in range(len(self.e))]
        self.g = [self._shift(tpost, i, True) for i in self.th]

    def nusselt(self, T, u):
        uh = u[0] if self.side else u[-1]
        return float(1.0 + self.L * (uh * T).mean() / self.alpha)


def _r16(t):
    """The BF16 rounding that the interface prescribes for a tensor."""
    return t.float().to(torch.bfloat16).double()


def _forward(ws, bs, x):
    """Outputs and BF16 activations of the network's layers, from FP64 weights."""
    acts, ys = [x], []
    for k, (w, b) in enumerate(zip(ws, bs)):
        ys.append(F.conv2d(acts[-1], _r16(w), b, padding=1))
        acts.append(_r16(ys[-1].relu()))
    return acts, ys


def exact(case, seed):
    kind = case["kind"]
    if kind in ("cell", "monitor"):
        shape, side = (case["nx"], case["ny"], case["nz"]), case["walls"] == "side"
        T, u = _rolls(case["dim"], shape, seed, side)
        m = _Flow(case["dim"], shape, case["Ra"], case["Pr"], T, u, side, case["periodic"])
        for _ in range(case.get("steps", 0)):
            m.step()
        _, rho, T, _, u = m.macros()
        out = {"rho": rho, "ux": u[0], "uy": u[1], "uz": u[2] if case["dim"] == 3 else torch.zeros_like(T), "T": T}
        if kind == "monitor" or case["nu"]:
            out["nu"] = m.nusselt(T, u)
        if kind == "monitor":
            out["ekin"], out["mass"] = float((0.5 * rho * sum(v * v for v in u)).sum()), float(rho.sum())
        return out
    if kind == "ensemble":
        got = {"T": [], "ux": [], "uy": []}
        nus = []
        for n, Ra, Pr, s in _members(case):
            T, u = _rolls(2, (n, n, 1), int(seed) * 1000 + s)
            m = _Flow(2, (n, n, 1), Ra, Pr, T, u, False, 0)
            for _ in range(case["steps"]):
                m.step()
            _, _, T, _, u = m.macros()
            nus.append(m.nusselt(T, u))
            for k, v in (("T", T), ("ux", u[0]), ("uy", u[1])):
                got[k].append(v.reshape(-1))
        return dict({k: torch.cat(v) for k, v in got.items()}, nu=torch.tensor(nus, dtype=torch.float64))
    if kind == "train":
        x16, tgt = _train_data(case, seed)
        net = _net(seed)
        ws, bs = [w.double() for w in net.w], [b.double() for b in net.b]
        acts, ys = _forward(ws, bs, x16.double())
        diff = ys[-1] - tgt.double()
        g = 2.0 * diff / diff.numel()
        gw, gb = [None] * len(ws), [None] * len(ws)
        for k in range(len(ws) - 1, -1, -1):
            gw[k] = torch.nn.grad.conv2d_weight(acts[k], ws[k].shape, _r16(g), padding=1)
            gb[k] = g.sum((0, 2, 3))
            if k > 0:
                g = torch.nn.grad.conv2d_input(acts[k].shape, _r16(ws[k]), _r16(g), padding=1) * (ys[k - 1] > 0)
        c1, c2 = 1.0 - 0.9 ** (net.t + 1), 1.0 - 0.999 ** (net.t + 1)

        def adam(p, d, m, v):
            m, v = 0.9 * m.double() + 0.1 * d, 0.999 * v.double() + 0.001 * d * d
            return p - 2e-3 * (m / c1) / ((v / c2).sqrt() + 1e-8)

        return {"y": ys[-1], "loss": (diff * diff).mean().reshape(1), "gw": gw, "gb": gb,
                "w": [adam(p, d, m, v) for p, d, m, v in zip(ws, gw, net.mw, net.vw)],
                "b": [adam(p, d, m, v) for p, d, m, v in zip(bs, gb, net.mb, net.vb)]}
    if kind == "layer":
        x, wt, b, dy = _layer_data(case, seed)
        y = F.conv2d(x.double(), _r16(wt), b.double(), padding=1)
        return {"y": y, "act": y.relu(),
                "dx": torch.nn.grad.conv2d_input(x.shape, _r16(wt), _r16(dy), padding=1),
                "dw": torch.nn.grad.conv2d_weight(x.double(), wt.shape, _r16(dy), padding=1),
                "db": dy.double().sum((0, 2, 3))}
    net, n = _net(seed), case["fine"]
    x = torch.tensor(surrogate.features(case["Ra"], case["Pr"], fine=n)[None], device="cuda")
    _, ys = _forward([w.double() for w in net.w], [b.double() for b in net.b], _r16(x))
    c = ys[-1][0]
    up = F.interpolate(c[None], size=(n, n), mode="bilinear", align_corners=True)[0]
    T, ux, uy = up[0].clamp(-0.5, 0.5), up[1] * U_FF, up[2] * U_FF
    m = _Flow(2, (n, n, 1), case["Ra"], case["Pr"], T, [ux, uy], False, 0)
    _, rho, T, _, u = m.macros()
    return {"coarse": c, "fields": {"rho": rho, "ux": u[0], "uy": u[1], "uz": torch.zeros_like(T), "T": T}}
