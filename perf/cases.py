"""What is measured of this library: the calls its users make, at the sizes they make them.

A case is one of these uses ("use"):

  steps   a context that is kept: the state goes in from device memory, a number of steps at the
          CFL step size is taken, the state comes out into device memory
  host    the same for a caller whose states live in pinned host memory: one step per call
  static  cr_step_static: one step of a given size for a caller that may not allocate
  batch   an ensemble of small problems advanced together with the learned blending coefficient
  train   training of the blending network on harvested samples

and "flow" names the initial data (the recipes of this repository's tests and benchmark).
"""
import math

import numpy as np
import torch

from paper_2502_07517_gb300 import crkfr

DEV = "cuda"
NVAR = {"linadv": 1, "euler1d": 3, "euler2d": 4, "tenmoment": 6}
EQ_OF = {"advection": "linadv", "riemann": "euler1d", "vortex": "euler2d", "box": "euler2d",
         "taylor": "euler2d", "voronoi": "tenmoment"}
LIMITED = frozenset({"blend", "mh", "flux", "scaling", "traces"})
SIDES = ("x-", "x+", "y-", "y+")


def _steps(name, flow, nx, ny, degree, steps, precision="fp64", alpha="indicator", diss="D2", central="EA",
           use="steps"):
    c = {"use": use, "flow": flow, "nx": nx, "ny": ny, "degree": degree, "steps": steps, "precision": precision,
         "alpha": alpha, "diss": diss, "central": central}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest run: a convergence or teaching study in 1D, hundreds of tiny steps
        _steps("advection-64", "advection", 64, 1, 3, 200),
        # a 1D shock tube at production resolution: still launch and latency bound
        _steps("riemann-4000", "riemann", 4000, 1, 4, 32),
        # one step inside a host program that owns all device memory: a ragged mesh
        _steps("static-61x59", "vortex", 61, 59, 4, 1, use="static"),
        # a caller with its states in host memory, one step per call
        _steps("host-256", "vortex", 256, 256, 4, 1, use="host"),
        # the flagship run and its form with FP32 bulk arithmetic
        _steps("vortex-512", "vortex", 512, 512, 4, 4),
        _steps("vortex-512-fp32", "vortex", 512, 512, 4, 8, precision="fp32"),
        # shocks in a walled box, the blending coefficient from the network
        _steps("box-256-fp32-net", "box", 256, 256, 4, 8, precision="fp32", alpha="net"),
        # ten-moment plasma with its source, in FP64 and, on a ragged mesh, in FP32 bulk
        _steps("voronoi-256", "voronoi", 256, 256, 3, 4),
        _steps("voronoi-211x173-fp32", "voronoi", 211, 173, 3, 8, precision="fp32"),
        # Rayleigh-Taylor: walls, given states with the HLLC flux, gravity
        _steps("taylor-64x256", "taylor", 64, 256, 3, 8),
        # an ensemble of small problems of uneven size and degree
        {"name": "ensemble-24", "use": "batch", "count": 24, "nmin": 32, "nmax": 128, "steps": 4},
        # training the network on samples harvested from runs
        {"name": "train-16", "use": "train", "nin": 16, "samples": 50000, "batch": 512, "epochs": 2},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    use = rng.choice(["1d", "1d", "2d", "2d", "2d", "2d", "host", "static", "batch", "train"])
    if use == "1d":
        if rng.random() < 0.4:
            return _steps("", "advection", _log_int(rng, 16, 1024), 1, rng.randint(1, 4), rng.randint(50, 400),
                          diss=rng.choice(["D2", "D1"]))
        return _steps("", "riemann", _log_int(rng, 100, 20000), 1, rng.randint(3, 4), rng.randint(8, 48),
                      precision=rng.choice(["fp64", "fp32"]), alpha=rng.choice(["indicator", "indicator", "net"]))
    if use == "2d":
        flow = rng.choice(["vortex", "vortex", "box", "voronoi", "taylor"])
        nx = _log_int(rng, 24, 440)
        ny = min(440, max(24, int(nx * rng.uniform(0.6, 1.6))))
        opt = {"precision": rng.choice(["fp64", "fp32"]), "alpha": rng.choice(["indicator", "indicator", "net"])}
        if flow == "vortex":
            opt.update(diss=rng.choice(["D2", "D2", "D1", "DCSX"]), central=rng.choice(["EA", "EA", "AE"]))
        if flow == "voronoi":
            nx, ny = min(nx, 256), min(ny, 256)
        degree = rng.choice([2, 3, 3, 4, 4, 4])
        if opt["precision"] == "fp32":  # built for degrees 3 and 4, the ten-moment equations for 3
            degree = 3 if flow == "voronoi" else max(3, degree)
        return _steps("", flow, nx, ny, degree, rng.randint(1, 4), **opt)
    if use == "host":
        return _steps("", "vortex", _log_int(rng, 48, 256), _log_int(rng, 48, 256), rng.randint(3, 4), 1, use="host",
                      precision=rng.choice(["fp64", "fp64", "fp32"]))
    if use == "static":
        return _steps("", rng.choice(["vortex", "voronoi"]), _log_int(rng, 8, 48), _log_int(rng, 8, 48), rng.randint(2, 4), 1,
                      use="static")
    if use == "batch":
        return {"use": "batch", "count": rng.randint(6, 32), "nmin": rng.randint(16, 40), "nmax": rng.randint(48, 128),
                "steps": rng.randint(1, 5)}
    return {"use": "train", "nin": rng.choice([5, 16, 25]), "samples": _log_int(rng, 8000, 60000),
            "batch": rng.choice([256, 512, 1024, 3000]), "epochs": rng.randint(1, 2)}


# --------------------------------------------------------------------- inputs
def _nodes(N):
    x, w = np.polynomial.legendre.leggauss(N + 1)
    return 0.5 * (x + 1.0), 0.5 * w


def _problem(flow, nx, ny, degree):
    """The problem as the binding's desc_from_problem takes it."""
    p = dict(dim=2, nx=nx, ny=ny, x0=0.0, x1=1.0, y0=0.0, y1=1.0, bc_x="periodic", bc_y="periodic", degree=degree,
             equation="euler", gamma=1.4, adv=(1.0, 0.0), source=None, limiter=LIMITED)
    if flow == "advection":
        p.update(dim=1, ny=1, equation="linadv", limiter=frozenset())
    elif flow == "riemann":
        p.update(dim=1, ny=1, bc_x="outflow")
    elif flow in ("vortex", "box"):
        p.update(x0=-5.0, x1=5.0, y0=-5.0, y1=5.0)
        if flow == "box":
            p.update(bc_x="wall", bc_y="wall")
    elif flow == "voronoi":
        p.update(equation="tenmoment", source=dict(amp=25.0, k=200.0, cx=0.5, cy=0.5))
    elif flow == "taylor":
        g = 5.0 / 3.0
        p.update(gamma=g, x1=0.25, bc_x="wall", bc_y="dirichlet", bc_flux="hllc", source=dict(gravity=(0.0, 1.0)),
                 bc_state={"y-": [2.0, 0.0, 0.0, 1.0 / (g - 1.0)], "y+": [1.0, 0.0, 0.0, 2.5 / (g - 1.0)]})
    return p


def _euler(rho, v, p, gamma):
    kin = 0.5 * rho * sum(x * x for x in v)
    return torch.stack([rho] + [rho * x for x in v] + [p / (gamma - 1.0) + kin])


def _state(prob, flow, seed):
    """The initial state [M][Ne][Np] on the GPU: this repository's recipes, from the seed."""
    rng = np.random.default_rng(seed)
    nx, ny, n, dim = prob["nx"], prob["ny"], prob["degree"] + 1, prob["dim"]
    xi = torch.tensor(_nodes(prob["degree"])[0], dtype=torch.float64, device=DEV)
    dx, dy = (prob["x1"] - prob["x0"]) / nx, (prob["y1"] - prob["y0"]) / ny
    at = lambda k, h, a: a + (torch.arange(k, dtype=torch.float64, device=DEV)[:, None] + xi) * h  # noqa: E731
    one = torch.ones((ny, nx, n if dim == 2 else 1, n), dtype=torch.float64, device=DEV)
    x = at(nx, dx, prob["x0"])[None, :, None, :] * one
    y = at(ny, dy, prob["y0"])[:, None, :, None] * one if dim == 2 else 0.0 * one
    ex = torch.arange(nx, device=DEV)[None, :, None, None] + torch.zeros_like(one, dtype=torch.long)
    ey = torch.arange(ny, device=DEV)[:, None, None, None] + torch.zeros_like(ex)
    if flow == "advection":
        k, phase = int(rng.integers(1, 4)), rng.uniform(0.0, 2.0 * math.pi)
        u = torch.sin(2.0 * math.pi * k * x + phase)[None]
    elif flow == "riemann":
        while True:  # two states that leave no vacuum between them
            rho = np.exp(rng.uniform(math.log(0.1), math.log(10.0), 2))
            vel = rng.uniform(-2.0, 2.0, 2)
            p = np.exp(rng.uniform(math.log(0.01), math.log(1000.0), 2))
            if vel[1] - vel[0] < 5.0 * np.sqrt(1.4 * p / rho).sum():
                break
        pick = lambda a: torch.where(ex >= nx // 2, float(a[1]), float(a[0])) * one  # noqa: E731
        u = _euler(pick(rho), [pick(vel)], pick(p), prob["gamma"])
    elif flow in ("vortex", "box"):
        g, beta = prob["gamma"], 5.0
        r2 = x * x + y * y
        rho = (1.0 - beta ** 2 * (g - 1.0) / (8.0 * g * math.pi ** 2) * torch.exp(1.0 - r2)) ** (1.0 / (g - 1.0))
        swirl = beta / (2.0 * math.pi) * torch.exp(0.5 * (1.0 - r2))
        v, p = [1.0 - y * swirl, 1.0 + x * swirl], rho ** g
        if flow == "vortex":  # a seeded 1% density perturbation of 8 periodic modes
            m, k, a, ph = rng.integers(1, 9, 8), rng.integers(1, 9, 8), rng.uniform(0.5, 1.0, 8), rng.uniform(0.0, 2.0 * math.pi, 8)
            pert = sum(float(a[i]) * torch.sin(2.0 * math.pi * (int(m[i]) * x + int(k[i]) * y) / 10.0 + float(ph[i])) for i in range(8))
            rho = rho * (1.0 + 0.01 * pert / pert.abs().max())
        else:  # a seeded planar jump, a stripe of half the domain
            rs, ps, along_x = rng.uniform(0.5, 5.0, 2), rng.uniform(0.1, 10.0, 2), bool(rng.integers(0, 2))
            e, k = (ex, nx) if along_x else (ey, ny)
            lo = int(rng.integers(k // 8, 3 * k // 8 + 1))
            inside = (e >= lo) & (e < lo + k // 2)
            rho = rho * torch.where(inside, float(rs[1]), float(rs[0]))
            p = p * torch.where(inside, float(ps[1]), float(ps[0]))
        u = _euler(rho, v, p, g)
    elif flow == "voronoi":  # piecewise constant by the seeded Voronoi cell of the element's centre
        sites, cells = torch.tensor(rng.uniform(0.0, 1.0, (16, 2)), device=DEV), 16
        rho, v = np.exp(rng.uniform(math.log(0.1), math.log(10.0), cells)), rng.uniform(-1.0, 1.0, (cells, 2))
        lam, ang = np.exp(rng.uniform(math.log(0.01), math.log(10.0), (cells, 2))), rng.uniform(0.0, math.pi, cells)
        c, s = np.cos(ang), np.sin(ang)
        p11, p22, p12 = c * c * lam[:, 0] + s * s * lam[:, 1], s * s * lam[:, 0] + c * c * lam[:, 1], c * s * (lam[:, 0] - lam[:, 1])
        per = np.stack([rho, rho * v[:, 0], rho * v[:, 1], 0.5 * p11 + 0.5 * rho * v[:, 0] ** 2,
                        0.5 * p12 + 0.5 * rho * v[:, 0] * v[:, 1], 0.5 * p22 + 0.5 * rho * v[:, 1] ** 2])
        cx = (torch.arange(nx, dtype=torch.float64, device=DEV) + 0.5) / nx
        cy = (torch.arange(ny, dtype=torch.float64, device=DEV) + 0.5) / ny
        ax, ay = (cx[None, :, None] - sites[:, 0]).abs(), (cy[:, None, None] - sites[:, 1]).abs()
        cell = (torch.minimum(ax, 1.0 - ax) ** 2 + torch.minimum(ay, 1.0 - ay) ** 2).argmin(-1)
        u = torch.tensor(per, device=DEV)[:, cell][..., None, None] * one
    else:  # Rayleigh-Taylor: heavy over light, seeded amplitude and wave number of the interface's motion
        g, low = prob["gamma"], ey * 2 < ny
        rho, p = torch.where(low, 2.0, 1.0) * one, torch.where(low, 2.0 * y + 1.0, y + 1.5)
        amp, k = 0.025 * rng.uniform(0.5, 1.5), int(rng.integers(1, 4))
        v2 = -amp * torch.sqrt(g * p / rho) * torch.cos(8.0 * math.pi * k * x)
        u = _euler(rho, [0.0 * one, v2], p, g)
    return u.reshape(u.shape[0], nx * ny, -1).contiguous()


def _alpha_from_energies(e, dim, N):
    """The smoothness indicator's alpha (before neighbour smoothing) from modal energies [..., q, p]."""
    i = torch.arange(N + 1, device=e.device)
    mx = torch.maximum(i[None, :], i[:, None] * (1 if dim == 2 else 0))[: e.shape[-2]]
    total = e.sum((-2, -1))
    low = (e * (mx <= N - 1)).sum((-2, -1))
    zero = torch.zeros_like(total)
    r = torch.where(total > 0, (e * (mx == N)).sum((-2, -1)) / total, zero)
    if N >= 2:
        r = torch.maximum(r, torch.where(low > 0, (e * (mx == N - 1)).sum((-2, -1)) / low, zero))
    T, s = 0.5 * 10.0 ** (-1.8 * (N + 1.0) ** 0.25), math.log((1.0 - 1e-4) / 1e-4)
    a = 1.0 / (1.0 + torch.exp(-s / T * (r - T)))
    return torch.where(a < 1e-3, 0.0, torch.where(a > 1.0 - 1e-3, 1.0, a)).to(e.dtype)


def _samples(nin, count, seed, dev):
    """Encoded modal energies as runs give them, from smooth to troubled elements, and their alpha."""
    dim = 2 if nin in (9, 16, 25) else 1
    n = int(round(math.sqrt(nin))) if dim == 2 else nin
    g = torch.Generator().manual_seed(seed)
    q = torch.arange(n if dim == 2 else 1)[:, None] + torch.arange(n)[None, :]
    decay = 0.3 + 11.7 * torch.rand((count, 1, 1), generator=g, dtype=torch.float64)
    m = torch.exp(-0.5 * decay * q + 0.7 * torch.randn((count,) + tuple(q.shape), generator=g, dtype=torch.float64))
    e = m * m
    e[:, 0, 0] *= 10.0 ** (2.0 * torch.rand(count, generator=g, dtype=torch.float64))
    e = e / e.sum((1, 2), keepdim=True)
    a = _alpha_from_energies(e, dim, n - 1)
    x = torch.log10(e + 1e-10) / 10.0 + 1.0
    return x.reshape(count, nin).float().to(dev), a.float().to(dev)


def _forward(p, x, nin):
    """The network's output logit; p [W1 32 x nin, b1, W2 32 x 32, b2, w3, b3]."""
    w1, b1, w2, b2, w3, b3 = torch.split(p, [32 * nin, 32, 1024, 32, 32, 1])
    h = torch.relu(x @ w1.view(32, nin).T + b1)
    h = torch.relu(h @ w2.view(32, 32).T + b2)
    return h @ w3 + b3


def _adam(p, x, t, order, batch, epochs, lr):
    """Adam on the cross-entropy over minibatches of order(epoch); the parameters and the last epoch's loss."""
    m, v, k, nin = torch.zeros_like(p), torch.zeros_like(p), 0, x.shape[1]
    for ep in range(epochs):
        idx, losses = order(ep), []
        for b in range(0, len(idx), batch):
            q = p.clone().requires_grad_(True)
            z, tt = _forward(q, x[idx[b:b + batch]], nin), t[idx[b:b + batch]]
            loss = (tt * torch.nn.functional.softplus(-z) + (1.0 - tt) * torch.nn.functional.softplus(z)).mean()
            g, = torch.autograd.grad(loss, q)
            losses.append(loss.detach())
            k += 1
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            p = p - lr * (m / (1.0 - 0.9 ** k)) / (torch.sqrt(v / (1.0 - 0.999 ** k)) + 1e-8)
    return p, torch.stack(losses).mean()


_NETS = {}


def _net(nin):
    """Parameters of a network that imitates the indicator (trained once on the host, the same everywhere)."""
    if nin not in _NETS:
        threads = torch.get_num_threads()
        torch.set_num_threads(1)
        x, t = _samples(nin, 8192, 7, "cpu")
        p = torch.from_numpy(np.random.default_rng(1).normal(0.0, 0.2, 32 * nin + 1121))
        order = lambda ep: torch.randperm(8192, generator=torch.Generator().manual_seed(ep))  # noqa: E731
        p, _ = _adam(p, x.double(), t.double(), order, 256, 12, 4e-3)
        torch.set_num_threads(threads)
        _NETS[nin] = p.float().numpy()
    return _NETS[nin]


def _ensemble(case, seed):
    rng = np.random.default_rng(seed)
    sides = np.random.default_rng(case["count"] * 1000 + case["nmax"]).integers(case["nmin"], case["nmax"] + 1, case["count"])
    degrees = 3 + np.arange(case["count"]) % 2
    return [(_problem("box", int(n), int(n), int(N)) | dict(bc_x="periodic", bc_y="periodic"), int(rng.integers(1 << 30)))
            for n, N in zip(sides, degrees)]


def _desc(prob, case):
    mode = crkfr.CR_ALPHA_MLP if case["alpha"] == "net" else crkfr.CR_ALPHA_INDICATOR
    diss = {"D2": crkfr.CR_DISS_D2, "D1": crkfr.CR_DISS_D1, "DCSX": crkfr.CR_DISS_DCSX}[case["diss"]]
    return crkfr.desc_from_problem(prob, precision=crkfr.CR_FP32_BULK if case["precision"] == "fp32" else crkfr.CR_FP64,
                                   alpha_mode=mode, dissipation=diss,
                                   central=crkfr.CR_CENTRAL_AE if case["central"] == "AE" else crkfr.CR_CENTRAL_EA)


def _context(prob, case):
    ctx = crkfr.cr_init_mesh(_desc(prob, case))
    if case["alpha"] == "net":
        crkfr.cr_mlp_load(ctx, _net((prob["degree"] + 1) ** prob["dim"]))
    return ctx


def _static_dt(prob):
    """A step size of about half the CFL limit of the recipes' largest wave speeds."""
    vmax = 3.5 if prob["equation"] == "euler" else 19.0
    return 0.03 / (vmax * (prob["nx"] / (prob["x1"] - prob["x0"]) + prob["ny"] / (prob["y1"] - prob["y0"])))


# ------------------------------------------------------------------ the calls
def prepare(case, seed):
    if case["use"] == "train":
        x, t = _samples(case["nin"], case["samples"], seed, DEV)
        p = torch.from_numpy(np.random.default_rng(seed).normal(0.0, 0.2, 32 * case["nin"] + 1121).astype(np.float32)).to(DEV)
        return {"case": case, "x": x, "t": t, "p": p, "seed": seed}
    if case["use"] == "batch":
        c = {"precision": "fp32", "alpha": "net", "diss": "D2", "central": "EA"}
        probs = _ensemble(case, seed)
        ctxs = [_context(p, c) for p, _ in probs]
        u = [_state(p, "box", s) for p, s in probs]
        b = crkfr.cr_batch_init(ctxs)
        crkfr.cr_batch_config(b, 256, crkfr.CR_BATCH_PHASES)  # what the autotuner picks for small meshes
        return {"case": case, "ctxs": ctxs, "u": u, "out": [torch.empty_like(x) for x in u], "batch": b}
    prob = _problem(case["flow"], case["nx"], case["ny"], case["degree"])
    u = _state(prob, case["flow"], seed)
    if case["use"] == "static":
        return {"case": case, "desc": _desc(prob, case), "u": u, "out": torch.empty_like(u), "dt": _static_dt(prob)}
    ctx = _context(prob, case)
    if case["use"] == "host":
        u = u.cpu().pin_memory()
        return {"case": case, "ctx": ctx, "u": u, "out": torch.empty(u.shape, dtype=u.dtype).pin_memory()}
    return {"case": case, "ctx": ctx, "u": u, "out": torch.empty_like(u)}


def run(s):
    case = s["case"]
    if case["use"] == "train":
        p = s["p"].clone()
        loss = crkfr.cr_mlp_train(case["nin"], p, s["x"], s["t"], batch=case["batch"], epochs=case["epochs"], lr=3e-3,
                                  seed=s["seed"])
        return {"params": p, "loss": loss}
    if case["use"] == "batch":
        for ctx, u in zip(s["ctxs"], s["u"]):
            crkfr.cr_set_state(ctx, u)
        crkfr.cr_batch_step(s["batch"], case["steps"])
        for ctx, out in zip(s["ctxs"], s["out"]):
            crkfr.cr_get_state(ctx, out)
        return s["out"]
    if case["use"] == "static":
        crkfr.cr_step_static(s["desc"], s["u"], s["out"], s["dt"])
        return s["out"]
    if case["use"] == "host":
        crkfr.cr_set_state(s["ctx"], s["u"].numpy())
        t, n = crkfr.cr_step_get(s["ctx"], 1, 1e300, s["out"])
        return {"u": s["out"], "t": t, "steps": n}
    crkfr.cr_set_state(s["ctx"], s["u"])
    t, n = crkfr.cr_step(s["ctx"], case["steps"], 1e300)
    return {"u": crkfr.cr_get_state(s["ctx"], s["out"]), "t": t, "steps": n}


def work(case):
    if case["use"] == "train":
        mac = 32 * case["nin"] + 1024 + 32  # per sample: forward, weight gradients, backward through two layers
        return {"bytes": 4 * case["samples"] * (case["nin"] + 1) * case["epochs"],
                "flops": case["samples"] * case["epochs"] * (2 * mac + 2 * mac + 2 * 1056)}
    if case["use"] == "batch":
        parts = [_flops("euler2d", p["degree"]) + (p["nx"] * p["ny"] * (p["degree"] + 1) ** 2,) for p, _ in _ensemble(case, 0)]
        return {"bytes": sum(2 * 8 * 4 * n for _, n in parts), "flops": case["steps"] * sum(f * n for f, n in parts)}
    eq, N = EQ_OF[case["flow"]], case["degree"]
    per = _flops(eq, N, limited=case["flow"] != "advection")[0]
    points = case["nx"] * case["ny"] * (N + 1) ** (2 if case["ny"] > 1 else 1)
    return {"bytes": 2 * 8 * NVAR[eq] * points, "flops": case["steps"] * per * points}


def _flops(eq, N, limited=True):
    """Flops per solution point and step, add, multiply, divide and square root one each, an FMA two."""
    dim = 2 if eq in ("euler2d", "tenmoment") else 1
    M, fl, sp, c2 = {"linadv": (1, 1, 1, 0), "euler1d": (3, 10, 10, 5), "euler2d": (4, 14, 12, 7), "tenmoment": (6, 24, 8, 19)}[eq]
    n = N + 1
    slots = 2 * dim * n ** (dim - 1) / n ** dim  # face nodes per solution point
    S, na, nb = {1: (2, 1, 1), 2: (3, 2, 2), 3: (4, 3, 4), 4: (6, 12, 5)}[N]
    f = na * M * 2 + S * dim * fl + nb * dim * M * 2 + S * M * dim * 2 * n  # stages, averages, derivatives
    f += nb * slots * (M * 2 * n + fl + 4 * M) + slots * sp  # face traces, their fluxes and averages
    f += slots / 2 * (7 * M) + dim * M * 4  # high-order interface flux and its terms of the update
    if limited:
        f += dim * M * 9 + 4 * dim * M + 2 * dim * fl + 7 * dim * M + 4 * dim * c2  # MUSCL-Hancock
        f += (dim * N / n + slots / 2) * (2 * fl + 2 * sp + 5 * M) + dim * M * 3  # low-order fluxes
        f += slots / 2 * 8 * (2 * M + c2) + slots * M * 2 * n + (1 + slots) * c2 + 2 * M + 2 * n * dim + 8  # limiters, indicator
    return (f,)


# ------------------------------------------------- the method in 64 bits, for exact()
def _lagrange(N):
    xi, w = _nodes(N)
    n = N + 1
    lag = lambda j, x: np.prod([(x - xi[m]) / (xi[j] - xi[m]) for m in range(n) if m != j])  # noqa: E731
    D = np.zeros((n, n))
    for j in range(n):
        for i in range(n):
            if i != j:
                D[i, j] = np.prod([(xi[i] - xi[m]) for m in range(n) if m not in (i, j)]) / np.prod([(xi[j] - xi[m]) for m in range(n) if m != j])
        D[j, j] = sum(1.0 / (xi[j] - xi[m]) for m in range(n) if m != j)
    return xi, w, np.array([lag(j, 0.0) for j in range(n)]), np.array([lag(j, 1.0) for j in range(n)]), D


TABLEAU = {
    1: ([[], [1 / 2]], [0, 1]),
    2: ([[], [1 / 3], [0, 2 / 3]], [1 / 4, 0, 3 / 4]),
    3: ([[], [1 / 2], [0, 1 / 2], [0, 0, 1]], [1 / 6, 1 / 3, 1 / 3, 1 / 6]),
    4: ([[], [1 / 4], [1 / 8, 1 / 8], [0, -1 / 2, 1], [3 / 16, 0, 0, 9 / 16], [-3 / 7, 2 / 7, 12 / 7, -12 / 7, 8 / 7]],
        [7 / 90, 0, 32 / 90, 12 / 90, 32 / 90, 7 / 90]),
}


def _cfl(N, d1):
    """The largest step per cell at which the linear scheme's amplification stays within 1 + 1e-4."""
    xi, w, l0, l1, D = _lagrange(N)
    gL, gR = -l0 / w, l1 / w
    ph = np.exp(-1j * np.linspace(0.0, 2.0 * math.pi, 721))[:, None, None]

    def growth(nu):
        T, Dm, fact = np.zeros_like(D), np.eye(N + 1), 1.0
        for m in range(N + 1):
            fact *= m + 1
            T += (-nu) ** m / fact * Dm
            Dm = Dm @ D
        V = np.eye(N + 1) if d1 else T
        A0 = D @ T + 0.5 * np.outer(gR, l1 @ V - l1 @ T) - 0.5 * np.outer(gL, l0 @ T + l0 @ V)
        Ap, A1 = 0.5 * np.outer(gR, l0 @ T - l0 @ V), 0.5 * np.outer(gL, l1 @ T + l1 @ V)
        G = np.eye(N + 1) - nu * (A0 + ph * A1 + ph.conj() * Ap)
        return np.abs(np.linalg.eigvals(G)).max()

    lo, hi = 0.0, 1.0
    for _ in range(40):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if growth(mid) <= 1.0 + 1e-4 else (lo, mid)
    return lo


class _Scheme:
    """The blended cRKFR step in torch float64; state [M, ny, nx, q, p]."""

    def __init__(self, prob, case, net=None):
        self.p, self.case, self.net = prob, case, net
        self.dim, self.N = prob["dim"], prob["degree"]
        self.eq = prob["equation"]
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=DEV)  # noqa: E731
        xi, w, l0, l1, D = _lagrange(self.N)
        self.np_w, self.w, self.l0, self.l1, self.D = w, t(w), t(l0), t(l1), t(D)
        self.h = [(prob["x1"] - prob["x0"]) / prob["nx"], (prob["y1"] - prob["y0"]) / prob["ny"]]
        X = np.concatenate([[xi[-1] - 1.0], xi, [1.0 + xi[0]]])
        self.ihm, self.ihp, self.ihc = t(1.0 / (X[1:-1] - X[:-2])), t(1.0 / (X[2:] - X[1:-1])), t(1.0 / (X[2:] - X[:-2]))
        cum = np.concatenate([[0.0], np.cumsum(w)])
        self.dm, self.dp = t(cum[:-1] - xi), t(cum[1:] - xi)
        leg = lambda j, x: np.polynomial.legendre.Legendre.basis(j)(2.0 * x - 1.0)  # noqa: E731
        self.V = t(np.array([[(2 * j + 1) * w[k] * leg(j, xi[k]) for k in range(self.N + 1)] for j in range(self.N + 1)]))
        self.cfl = _cfl(self.N, case["diss"] == "D1")
        self.lim = prob["limiter"]
        self.bc = [prob["bc_x"], prob["bc_y"]]
        src = prob["source"]
        self.src = None
        if src and "gravity" in src:
            self.src = [float(g) for g in src["gravity"]]
        elif src:
            n, nx, ny = self.N + 1, prob["nx"], prob["ny"]
            x = prob["x0"] + (torch.arange(nx, device=DEV)[:, None] + t(xi)) * self.h[0]
            y = prob["y0"] + (torch.arange(ny, device=DEV)[:, None] + t(xi)) * self.h[1]
            rx, ry = x[None, :, None, :] - src["cx"], y[:, None, :, None] - src["cy"]
            W = src["amp"] * torch.exp(-src["k"] * (rx * rx + ry * ry))
            self.src = [-2.0 * src["k"] * rx * W, -2.0 * src["k"] * ry * W]

    # ---- the equations
    def pressure(self, u):
        return (self.p["gamma"] - 1.0) * (u[-1] - 0.5 * sum(u[1 + d] ** 2 for d in range(self.dim)) / u[0])

    def flux(self, u, d):
        if self.eq == "linadv":
            return self.p["adv"][d] * u
        v = u[1 + d] / u[0]
        if self.eq == "euler":
            p = self.pressure(u)
            f = [u[1 + d]] + [u[1 + k] * v + (p if k == d else 0.0) for k in range(self.dim)] + [(u[-1] + p) * v]
            return torch.stack(f)
        v1, v2 = u[1] / u[0], u[2] / u[0]
        p11, p12, p22 = 2.0 * u[3] - u[1] * v1, 2.0 * u[4] - u[1] * v2, 2.0 * u[5] - u[2] * v2
        if d == 0:
            return torch.stack([u[1], p11 + u[1] * v1, p12 + u[1] * v2, (u[3] + p11) * v1,
                                u[4] * v1 + 0.5 * (p11 * v2 + p12 * v1), u[5] * v1 + p12 * v2])
        return torch.stack([u[2], p12 + u[1] * v2, p22 + u[2] * v2, u[3] * v2 + p12 * v1,
                            u[4] * v2 + 0.5 * (p12 * v2 + p22 * v1), (u[5] + p22) * v2])

    def speed(self, u, d):
        if self.eq == "linadv":
            return torch.full_like(u[0], abs(self.p["adv"][d]))
        v = u[1 + d] / u[0]
        if self.eq == "euler":
            return v.abs() + torch.sqrt((self.p["gamma"] * self.pressure(u) / u[0]).clamp_min(0.0))
        return v.abs() + torch.sqrt((3.0 * (2.0 * u[3 + 2 * d] - u[1 + d] * v) / u[0]).clamp_min(0.0))

    def second(self, u):
        if self.eq == "euler":
            return self.pressure(u)
        p11, p12, p22 = 2.0 * u[3] - u[1] ** 2 / u[0], 2.0 * u[4] - u[1] * u[2] / u[0], 2.0 * u[5] - u[2] ** 2 / u[0]
        return 0.5 * (p11 + p22) - torch.sqrt((0.5 * (p11 - p22)) ** 2 + p12 ** 2)

    def source(self, u):
        g1, g2 = self.src
        if self.eq == "euler":
            return torch.stack([0.0 * u[0], u[0] * g1, u[0] * g2, u[1] * g1 + u[2] * g2])
        return torch.stack([0.0 * u[0], -0.5 * u[0] * g1, -0.5 * u[0] * g2, -0.5 * u[1] * g1,
                            -0.25 * (u[2] * g1 + u[1] * g2), -0.5 * u[2] * g2])

    # ---- one-dimensional operators in direction d (0: p, 1: q)
    def mat(self, A, x, d):
        return x @ A.T if d == 0 else (x.transpose(-1, -2) @ A.T).transpose(-1, -2)

    def trace(self, l, x, d):
        return x @ l if d == 0 else x.transpose(-1, -2) @ l

    def vec(self, a, d):
        return a if d == 0 else a[:, None]

    def slope(self, u, d, beta):
        """minmod slopes of the node values, halo nodes from the neighbour elements."""
        ax, el = (-1, 2) if d == 0 else (-2, 1)
        first, last = u.narrow(ax, 0, 1), u.narrow(ax, self.N, 1)
        lo, hi = torch.roll(last, 1, el), torch.roll(first, -1, el)
        if self.bc[d] != "periodic":
            k = u.shape[el]
            lo = torch.cat([self.ghost(first.narrow(el, 0, 1), d, 0), lo.narrow(el, 1, k - 1)], el)
            hi = torch.cat([hi.narrow(el, 0, k - 1), self.ghost(last.narrow(el, k - 1, 1), d, 1)], el)
        um = torch.cat([lo, u.narrow(ax, 0, self.N)], ax)
        up = torch.cat([u.narrow(ax, 1, self.N), hi], ax)
        a = beta * self.vec(self.ihm, d) * (u - um)
        b = self.vec(self.ihc, d) * (up - um)
        c = beta * self.vec(self.ihp, d) * (up - u)
        small = torch.minimum(torch.minimum(a.abs(), b.abs()), c.abs())
        same = (torch.sign(a) == torch.sign(b)) & (torch.sign(a) == torch.sign(c))
        return torch.where(same, torch.sign(a) * small, torch.zeros_like(small))

    def ghost(self, u, d, side):
        """Ghost values of a boundary side for values u inside it (outflow: u itself)."""
        if self.bc[d] == "wall":
            s = torch.ones(u.shape[0], dtype=u.dtype, device=DEV)
            s[1 + d] = -1.0
            return u * s.view(-1, *[1] * (u.dim() - 1))
        if self.bc[d] == "dirichlet":
            g = torch.tensor(self.p["bc_state"][SIDES[2 * d + side]], dtype=u.dtype, device=DEV)
            return g.view(-1, *[1] * (u.dim() - 1)).expand_as(u)
        return u

    def sides(self, t0, t1, d, ghost):
        """Left and right values at the n + 1 faces of each line from the elements' two traces."""
        el = t0.dim() - 2 if d == 0 else t0.dim() - 3
        k = t0.shape[el]
        if self.bc[d] == "periodic":
            return torch.cat([t1.narrow(el, k - 1, 1), t1], el), torch.cat([t0, t0.narrow(el, 0, 1)], el)
        gl, gr = ghost(t0.narrow(el, 0, 1), 0), ghost(t1.narrow(el, k - 1, 1), 1)
        return torch.cat([gl, t1], el), torch.cat([t0, gr], el)

    def hllc(self, UL, UR, FL, FR, d):
        pl, pr, rl, rr = self.pressure(UL), self.pressure(UR), UL[0], UR[0]
        vl, vr, g = UL[1 + d] / rl, UR[1 + d] / rr, self.p["gamma"]
        cl, cr = torch.sqrt((g * pl / rl).clamp_min(0.0)), torch.sqrt((g * pr / rr).clamp_min(0.0))
        sl, sr = torch.minimum(vl - cl, vr - cr), torch.maximum(vl + cl, vr + cr)
        ss = (pr - pl + rl * vl * (sl - vl) - rr * vr * (sr - vr)) / (rl * (sl - vl) - rr * (sr - vr))

        def star(U, F, r, vn, p, sk):
            fac = r * (sk - vn) / (sk - ss)
            us = [fac * U[k] / r for k in range(U.shape[0])]
            us[0], us[1 + d] = fac, fac * ss
            us[-1] = fac * (U[-1] / r + (ss - vn) * (ss + p / (r * (sk - vn))))
            return F + sk * (torch.stack(us) - U)

        out = torch.where(ss >= 0.0, star(UL, FL, rl, vl, pl, sl), star(UR, FR, rr, vr, pr, sr))
        return torch.where(sl >= 0.0, FL, torch.where(sr <= 0.0, FR, out))

    def rusanov(self, L, R, d, lam=None):
        lam = torch.maximum(self.speed(L, d), self.speed(R, d)) if lam is None else lam
        return 0.5 * (self.flux(L, d) + self.flux(R, d)) - 0.5 * lam * (R - L)

    # ---- the blending coefficient
    def modal(self, u):
        x = u[0] if self.eq == "linadv" else u[0] * self.pressure(u) if self.eq == "euler" else \
            u[0] * 0.5 * (2.0 * u[3] - u[1] ** 2 / u[0] + 2.0 * u[5] - u[2] ** 2 / u[0])
        m = self.mat(self.V, x, 0)
        return (self.mat(self.V, m, 1) if self.dim == 2 else m) ** 2

    def raw_alpha(self, u):
        e = self.modal(u)
        a = _alpha_from_energies(e, self.dim, self.N)
        if self.net is not None:
            total = e.sum((-2, -1), keepdim=True)
            x = torch.log10(torch.where(total > 0, e / total, torch.zeros_like(e)) + 1e-10) / 10.0 + 1.0
            y = torch.sigmoid(_forward(self.net, x.reshape(-1, e.shape[-1] * e.shape[-2]), e.shape[-1] * e.shape[-2])).view_as(a)
            a = torch.where(y < 1e-3, 0.0, torch.where(y > 1.0 - 1e-3, 1.0, y)).to(u.dtype)
        return a

    def smooth(self, raw):
        a = raw
        for d in range(self.dim):
            el = 1 - d
            for s in (1, -1):
                r = torch.roll(raw, s, el)
                if self.bc[d] != "periodic":
                    r = r.clone()
                    r.select(el, 0 if s == 1 else r.shape[el] - 1).zero_()
                a = torch.maximum(a, 0.5 * r)
        return a

    def means(self, u):
        m = u @ self.w
        return m @ self.w if self.dim == 2 else m[..., 0]

    def dt(self, u):
        m = self.means(u)
        return 0.98 * self.cfl / float(sum(self.speed(m, d) / self.h[d] for d in range(self.dim)).max())

    # ---- one step
    def step(self, u, raw, dt):
        dim, N, w = self.dim, self.N, self.w
        A, b = TABLEAU[N]
        blend, limited = "blend" in self.lim, bool(self.lim)
        alpha = self.smooth(raw) if blend else torch.zeros_like(raw)
        al = alpha[:, :, None, None]
        stages, L, Fs = [], [], []
        for i in range(len(b)):
            ui = u - dt * sum(A[i][j] * L[j] for j in range(i)) if i else u
            f = [self.flux(ui, d) for d in range(dim)]
            r = sum(self.mat(self.D, f[d], d) / self.h[d] for d in range(dim))
            L.append(r - self.source(ui) if self.src else r)
            stages.append(ui)
            Fs.append(f)
        U = sum(b[i] * stages[i] for i in range(len(b)))
        F = [sum(b[i] * Fs[i][d] for i in range(len(b))) for d in range(dim)]
        P = u
        if self.src:
            P = P + dt * sum(b[i] * self.source(stages[i]) for i in range(len(b)))
        if limited:  # MUSCL-Hancock face states of the subcells
            beta = 2.0 - al
            fm, fp = [], []
            for d in range(dim):
                s = self.slope(u, d, beta)
                fm.append(u + self.vec(self.dm, d) * s)
                fp.append(u + self.vec(self.dp, d) * s)
            ev = sum(0.5 * dt * (self.flux(fp[d], d) - self.flux(fm[d], d)) / (self.vec(w, d) * self.h[d]) for d in range(dim))
            ok = torch.ones_like(u[0], dtype=torch.bool)
            for s in [x for pair in zip(fm, fp) for x in pair]:
                for x in (s, s - ev):
                    ok &= (x[0] > 0.0) & (self.second(x) > 0.0)
            fm = [torch.where(ok, x - ev, u) for x in fm]
            fp = [torch.where(ok, x - ev, u) for x in fp]
        new = P
        for d in range(dim):
            ax, el, h = (-1, 2, self.h[0]) if d == 0 else (-2, 1, self.h[1])
            l = (self.l0, self.l1)
            new = new - dt * (1.0 - al) * self.mat(self.D - torch.outer(self.l1 / w, self.l1) + torch.outer(self.l0 / w, self.l0), F[d], d) / h
            gh = lambda x, s: self.ghost(x, d, s)  # noqa: E731
            un = [self.trace(l[s], u, d) for s in (0, 1)]
            Ut = [self.trace(l[s], U, d) for s in (0, 1)]
            st = [[self.trace(l[s], x, d) for s in (0, 1)] for x in stages]
            if self.case["central"] == "AE":
                Ft = [self.trace(l[s], F[d], d) for s in (0, 1)]
            else:
                Ft = [sum(b[i] * self.flux(st[i][s], d) for i in range(len(b)) if b[i]) for s in (0, 1)]

            def ghost_flux(x, s):
                if self.bc[d] == "wall":
                    sg = -torch.ones(x.shape[0], dtype=x.dtype, device=DEV)
                    sg[1 + d] = 1.0
                    return x * sg.view(-1, *[1] * (x.dim() - 1))
                return self.flux(gh(x, s), d) if self.bc[d] == "dirichlet" else x

            FL, FR = self.sides(Ft[0], Ft[1], d, ghost_flux)
            nL, nR = self.sides(un[0], un[1], d, gh)
            UL, UR = self.sides(Ut[0], Ut[1], d, gh)
            lam = torch.maximum(self.speed(nL, d), self.speed(nR, d))
            if self.case["diss"] == "DCSX":
                diss = 0.0
                for i in range(len(b)):
                    if b[i]:
                        a, c = self.sides(st[i][0], st[i][1], d, gh)
                        diss = diss + 0.5 * b[i] * torch.maximum(self.speed(a, d), self.speed(c, d)) * (c - a)
            else:
                diss = 0.5 * lam * ((nR - nL) if self.case["diss"] == "D1" else (UR - UL))
            FH = 0.5 * (FL + FR) - diss
            hllc, out = self.bc[d] == "dirichlet", self.bc[d] == "outflow"
            el_f = FH.dim() - 2 if d == 0 else FH.dim() - 3
            k = FH.shape[el_f]

            def edges(x, y):
                """x inside, y at the two boundary faces."""
                return torch.cat([y.narrow(el_f, 0, 1), x.narrow(el_f, 1, k - 2), y.narrow(el_f, k - 1, 1)], el_f) if k > 2 else y

            if hllc:
                FH = edges(FH, self.hllc(UL, UR, FL, FR, d))
            elif out:
                FH = edges(FH, torch.cat([FR.narrow(el_f, 0, 1), FL.narrow(el_f, 1, k - 1)], el_f))
            Fn = FH
            if limited:
                bm, bp = fm[d].select(ax, 0), fp[d].select(ax, N)
                sL, sR = self.sides(bm, bp, d, gh)
                FLO = self.rusanov(sL, sR, d)
                if hllc:
                    FLO = edges(FLO, self.hllc(sL, sR, self.flux(sL, d), self.flux(sR, d), d))
                elif out:
                    inner = torch.cat([sR.narrow(el_f, 0, 1), sL.narrow(el_f, 1, k - 1)], el_f)
                    FLO = edges(FLO, self.flux(inner, d))
                a0 = alpha[:, :, None]
                aL, aR = self.sides(a0, a0, d, lambda x, s: x)
                af = (0.5 * (aL + aR))[None]
                Fn = (1.0 - af) * FH + af * FLO
                sub = self.rusanov(fp[d].narrow(ax, 0, N), fm[d].narrow(ax, 1, N), d)
                Fn = self.limit_flux(Fn, FLO, u, sub, dt, d, ax, el_f)
                zero = torch.zeros_like(u.narrow(ax, 0, 1))
                lo = (torch.cat([sub, zero], ax) - torch.cat([zero, sub], ax)) / (self.vec(w, d) * h)
                new = new - dt * al * lo
            k -= 1
            fl, fr = Fn.narrow(el_f, 0, k).unsqueeze(ax), Fn.narrow(el_f, 1, k).unsqueeze(ax)
            e0 = torch.zeros(N + 1, dtype=torch.float64, device=DEV)
            eN = e0.clone()
            e0[0], eN[N] = 1.0 / w[0], 1.0 / w[N]
            cR = (1.0 - al) * self.vec(self.l1 / w, d) + al * self.vec(eN, d)
            cL = -(1.0 - al) * self.vec(self.l0 / w, d) - al * self.vec(e0, d)
            new = new - dt / h * (fr * cR + fl * cL)
        return self.scale(new) if limited else new

    def limit_flux(self, F, FLO, u, sub, dt, d, ax, el):
        kappa = 0.5 if self.dim == 2 else 1.0
        k = F.shape[el]
        c0, c1 = dt / (kappa * self.np_w[0] * self.h[d]), dt / (kappa * self.np_w[-1] * self.h[d])
        base0, base1 = u.select(ax, 0) - c0 * sub.select(ax, 0), u.select(ax, self.N) + c1 * sub.select(ax, self.N - 1)
        if self.bc[d] == "periodic":
            bL, bR = torch.cat([base1.narrow(el, k - 2, 1), base1], el), torch.cat([base0, base0.narrow(el, 0, 1)], el)
            hasL = hasR = None
        else:
            bL, bR = torch.cat([base1.narrow(el, 0, 1), base1], el), torch.cat([base0, base0.narrow(el, k - 2, 1)], el)
            i = torch.arange(k, device=DEV).view([-1 if a == el - 1 else 1 for a in range(F.dim() - 1)])
            hasL, hasR = i > 0, i < k - 1
        theta = torch.ones_like(F[0])
        dead = torch.zeros_like(theta, dtype=torch.bool)
        for con in (lambda x: x[0], self.second):
            inf = torch.full_like(theta, math.inf)
            lowL, lowR = con(bL - c1 * FLO), con(bR + c0 * FLO)
            eps = 0.1 * torch.minimum(lowL if hasL is None else torch.where(hasL, lowL, inf), lowR if hasR is None else torch.where(hasR, lowR, inf))
            dead |= ~(eps > 0.0)
            Ft = theta * F + (1.0 - theta) * FLO
            tk = torch.ones_like(theta)
            for low, P, has in ((lowL, con(bL - c1 * Ft), hasL), (lowR, con(bR + c0 * Ft), hasR)):
                bad = P < eps if has is None else (P < eps) & has
                tk = torch.where(bad, torch.minimum(tk, (low - eps) / (low - P)), tk)
            theta = torch.where(dead, torch.zeros_like(theta), theta * tk)
        return theta * F + (1.0 - theta) * FLO

    def scale(self, u):
        """The scaling limiter on the nodes and the face traces of the elements that need it."""
        M, N = u.shape[0], self.N
        pts = [u.flatten(3)]
        for d in range(self.dim):
            pts += [self.trace(l, u, d).flatten(3) for l in (self.l0, self.l1)]
        pts = torch.cat(pts, -1).flatten(1, 2)
        ub = self.means(u).flatten(1, 2)
        e1, e2 = ub[0].clamp_max(1e-12), self.second(ub).clamp_max(1e-12)
        need = ((pts[0] < e1[:, None]) | ~(self.second(pts) >= e2[:, None])).any(1).nonzero()[:, 0]
        if not len(need):
            return u
        p, m, e1, e2 = pts[:, need].clone(), ub[:, need, None], e1[need, None], e2[need, None]
        rmin = p[0].min(1, keepdim=True).values
        th = torch.where(rmin < e1, (m[0] - e1) / (m[0] - rmin), torch.ones_like(rmin))
        p[0] = torch.where(rmin < e1, m[0] + th * (p[0] - m[0]), p[0])
        lo, hi = torch.zeros_like(p[0]), torch.ones_like(p[0])
        fine = self.second(p) >= e2
        for _ in range(50):
            mid = 0.5 * (lo + hi)
            good = self.second(m + mid * (p - m)) >= e2
            lo, hi = torch.where(good, mid, lo), torch.where(good, hi, mid)
        t2 = torch.where(fine, torch.ones_like(lo), lo).min(1, keepdim=True).values
        p = torch.where(t2 < 1.0, m + t2 * (p - m), p)
        out = u.flatten(3).flatten(1, 2).clone()
        out[:, need] = p[..., : out.shape[-1]]
        return out.view_as(u)

    def run(self, u, steps, dt=None):
        n, shape = self.N + 1, u.shape
        u = u.view(shape[0], self.p["ny"], self.p["nx"], n if self.dim == 2 else 1, n)
        t = 0.0
        for _ in range(steps):
            h = self.dt(u) if dt is None else dt
            u = self.step(u, self.raw_alpha(u), h)
            t += h
        return u.reshape(shape), t


def _shuffles(n, epochs, seed):
    """The seeded orders of the training samples: Fisher-Yates driven by splitmix64."""
    s, mask, orders = seed, (1 << 64) - 1, []
    for _ in range(epochs):
        perm = list(range(n))
        for i in range(n - 1, 0, -1):
            s = (s + 0x9e3779b97f4a7c15) & mask
            z = s
            z = ((z ^ (z >> 30)) * 0xbf58476d1ce4e5b9) & mask
            z = ((z ^ (z >> 27)) * 0x94d049bb133111eb) & mask
            j = (z ^ (z >> 31)) % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        orders.append(torch.tensor(perm, device=DEV))
    return orders


def _exact_net(nin):
    return torch.tensor(_net(nin)).to(torch.bfloat16).double().to(DEV)  # the library keeps the weights in BF16


def exact(case, seed):
    if case["use"] == "train":
        x, t = _samples(case["nin"], case["samples"], seed, DEV)
        p = torch.from_numpy(np.random.default_rng(seed).normal(0.0, 0.2, 32 * case["nin"] + 1121).astype(np.float32))
        orders = _shuffles(case["samples"], case["epochs"], seed)
        p, loss = _adam(p.double().to(DEV), x.double(), t.double(), lambda ep: orders[ep], case["batch"], case["epochs"], 3e-3)
        return {"params": p, "loss": float(loss)}
    if case["use"] == "batch":
        c = {"diss": "D2", "central": "EA"}
        return [_Scheme(p, c, _exact_net((p["degree"] + 1) ** 2)).run(_state(p, "box", s), case["steps"])[0]
                for p, s in _ensemble(case, seed)]
    prob = _problem(case["flow"], case["nx"], case["ny"], case["degree"])
    net = _exact_net((case["degree"] + 1) ** prob["dim"]) if case["alpha"] == "net" else None
    u = _state(prob, case["flow"], seed)
    scheme = _Scheme(prob, case, net)
    if case["use"] == "static":
        return scheme.run(u, 1, _static_dt(prob))[0]
    out, t = scheme.run(u, case["steps"])
    return {"u": out.cpu() if case["use"] == "host" else out, "t": t, "steps": None}
