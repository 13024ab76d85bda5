"""Workloads that stand for the use of this package, each through its public
Python entry points (``lbm.Lattice``, ``lbm.Batch``), with a plain 64-bit
torch evaluation of the same method beside it.

A lattice case is one job of a user's program: the state from a density and
velocity field, a run of time steps, then the populations and the
macroscopic fields read back.  The sizes are those of the paper's studies and
of this repository's benchmark: the 800-site shock tube, the 100^2 box of
the Hopf study, the 129^2 cavity of the stability study, the 257^2, 2049^2
and 4097^2 cavities, a batch of mixed cavities, and the gradient of the
513^2 cavity.  Runs are short pieces of the real ones, started from a smooth
recirculating flow under a moving lid (what such a run spends nearly all of
its steps in) whose modes come from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1110_0270_gb300 import lbm
from paper_1110_0270_gb300 import workloads as WL

BYTES = {"fp64": 8, "fp32": 4, "fp16_dev": 2, "bf16_dev": 2}
# arithmetic per site and step that the collision cannot do without
# (D2Q9; D1Q3 about a third): moments, equilibrium, relaxation, and for the
# limiters Delta S, for ELBM its root
FLOPS = {"lbgk": 110, "positivity": 120, "ehrenfest": 140, "median": 140, "mrt": 180, "mrt2": 130,
         "mrt_limiter": 140, "smooth": 250, "double_monotonic": 260, "ensemble": 260, "ensemble_lagged": 260,
         "threshold": 250, "elbm": 700}

# the limiters' parameters in the benchmark's variants
LIMITERS = {"smooth": dict(lim_alpha=40.0, lim_k=1.0), "double_monotonic": dict(lim_dst=2e-3, lim_k=1.5),
            "ensemble": dict(lim_alpha=1.0, lim_k=1.0), "ensemble_lagged": dict(lim_alpha=1.0, lim_k=1.0),
            "threshold": dict(lim_delta0=0.01)}


def _lattice(name, nx, ny, collision, precision, steps, bc="cavity", re=5000.0, lid=0.1, topk=64, equilibrium="poly",
             probe=False):
    c = dict(kind="lattice", nx=nx, ny=ny, collision=collision, precision=precision, steps=steps, bc=bc, re=re,
             lid=lid, topk=topk, equilibrium=equilibrium, probe=probe)
    return dict(c, name=name) if name else c


def _tube(name, nx, collision, precision, steps):
    c = dict(kind="tube", nx=nx, collision=collision, precision=precision, steps=steps, topk=4)
    return dict(c, name=name) if name else c


def listed():
    return [
        # Section 6's shock tube, the plain method and the entropic one: the
        # smallest lattice, a run of 400 steps as the paper plots it
        _tube("tube800_lbgk_f64", 800, "lbgk", "fp64", 400),
        _tube("tube800_elbm_f64", 800, "elbm", "fp64", 400),
        # Section 8's Hopf study: 100^2 box with diffusive walls, entropic
        # equilibria, median filter, the control point recorded every step
        _lattice("hopf100_median_f64", 100, 100, "median", "fp64", 400, bc="diffusive", re=7000.0,
                 equilibrium="entropic", probe=True),
        # Section 8's stability study: 129^2 cavity, at most nine Ehrenfest
        # steps per time step, FP64
        _lattice("stability129_ehrenfest_f64", 129, 129, "ehrenfest", "fp64", 400, topk=9),
        # the 257^2 cavity at Re 5000 in both full precisions
        _lattice("cavity257_ehrenfest_f32", 257, 257, "ehrenfest", "fp32", 400),
        _lattice("cavity257_mrt_f64", 257, 257, "mrt", "fp64", 400),
        # the bandwidth configuration, 4097^2 at Re 10000: the headline step
        # and the 16-bit storage of the same lattice
        _lattice("cavity4097_ehrenfest_f32", 4097, 4097, "ehrenfest", "fp32", 20, re=10000.0, lid=0.05),
        _lattice("cavity4097_lbgk_f16", 4097, 4097, "lbgk", "fp16_dev", 20, re=10000.0, lid=0.05),
        # ELBM in a flow that has left rest: every site solves for alpha
        _lattice("cavity2049_elbm_f32", 2049, 2049, "elbm", "fp32", 10, re=10000.0, lid=0.05),
        # a limiter of Section 4.4 that evaluates Delta S at every site
        _lattice("cavity2049_threshold_f32", 2049, 2049, "threshold", "fp32", 20, re=10000.0, lid=0.05),
        # the batched configuration: cavities of sides 64 to 768, LBGK, ELBM,
        # Ehrenfest and median in turn
        dict(kind="batch", name="batch32_mixed_f32", n=32, precision="fp32", steps=20, list_seed=0),
        # the gradient of the kinetic energy, Ehrenfest steps, checkpoints
        # every 100 steps
        dict(kind="adjoint", name="adjoint513_ehrenfest_f32", nx=513, ny=513, collision="ehrenfest",
             precision="fp32", T=400, K=100, re=1000.0, lid=0.1, topk=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case over the same ranges: tubes of 100 to 20000 sites, boxes
    of 48 to 400 sites a side (every boundary), planes up to 4097^2 in every
    storage format, batches and gradients."""
    kind = rng.choice(["tube", "box", "box", "plane", "plane", "batch", "adjoint"])
    if kind == "tube":
        return _tube(None, _log(rng, 100, 20000), rng.choice(["lbgk", "elbm", "ehrenfest", "median"]),
                     rng.choice(["fp64", "fp64", "fp32"]), 2 * rng.randint(50, 250))
    if kind == "box":
        bc = rng.choice(["cavity", "cavity", "diffusive", "periodic", "channel"])
        coll = rng.choice(["lbgk", "ehrenfest", "median", "mrt", "mrt_limiter", "elbm", "smooth", "threshold"])
        return _lattice(None, _log(rng, 48, 400), _log(rng, 48, 400), coll, rng.choice(["fp64", "fp32"]),
                        rng.randint(40, 300) if coll == "elbm" else rng.randint(100, 500), bc=bc,
                        re=float(_log(rng, 100, 5000)), topk=rng.choice([4, 9, 64]),
                        equilibrium=rng.choice(["poly", "entropic", "poly_std"]))
    if kind == "plane":
        prec = rng.choice(["fp32", "fp32", "fp16_dev", "bf16_dev", "fp64"])
        coll = rng.choice(["lbgk", "ehrenfest", "median", "positivity", "mrt", "mrt2", "mrt_limiter", "smooth",
                           "ensemble_lagged", "threshold", "elbm"])
        hi = 2049 if coll == "elbm" or prec == "fp64" else 4097
        return _lattice(None, _log(rng, 400, hi), _log(rng, 400, hi), coll, prec, rng.randint(4, 9), lid=0.05,
                        re=float(_log(rng, 1000, 10000)))
    if kind == "batch":
        return dict(kind="batch", n=rng.randint(8, 32), precision=rng.choice(["fp32", "fp32", "fp16_dev"]),
                    steps=2 * rng.randint(4, 10), list_seed=rng.randint(1, 10 ** 6))
    side = _log(rng, 65, 513)
    return dict(kind="adjoint", nx=side, ny=_log(rng, 65, 513),
                collision=rng.choice(["lbgk", "ehrenfest", "median", "positivity"]), precision="fp32",
                T=20 * rng.randint(5, 20), K=rng.choice([25, 50, 100]), re=1000.0, lid=0.1, topk=32)


# ----------------------------------------------------------------- inputs
def _config(case):
    if case["kind"] == "tube":
        cfg, _ = WL.shock_tube(case["nx"])
        return dict(cfg, collision=case["collision"], precision=case["precision"], topk=case["topk"], delta=1e-3)
    L = max(case["nx"], case["ny"]) - 1
    cfg = dict(lattice="D2Q9", nx=case["nx"], ny=case["ny"], bc=case.get("bc", "cavity"), lid_u=case["lid"],
               collision=case["collision"], precision=case["precision"], topk=case["topk"], delta=1e-3,
               equilibrium=case.get("equilibrium", "poly"), s_e=1.64, s_eps=1.64, s_q=1.2)
    nu = case["lid"] * L / case["re"]
    return dict(cfg, nu=nu, beta=1.0 / (6.0 * nu + 1.0), **LIMITERS.get(case["collision"], {}))


def _batch_configs(case):
    out = []
    for inst in WL.batched_cavities(n=case["n"], seed=case["list_seed"]):
        cfg, _ = WL.cavity(inst["side"], inst["re"], 0.1)
        out.append(dict(cfg, collision=inst["collision"], precision=case["precision"], topk=64, delta=1e-3,
                        beta=1.0 / (6.0 * cfg["nu"] + 1.0), equilibrium="poly"))
    return out


def _flow(cfg, seed):
    """Density and velocity [ny][nx] (float64, on the GPU): the jump of the
    tube with a little noise, or a recirculating flow of a few seeded modes,
    at rest on resting walls and moving with the lid in a layer below it."""
    ny, nx = cfg["ny"], cfg["nx"]
    rng = np.random.default_rng(seed)
    dev = torch.device("cuda")
    if cfg["lattice"] == "D1Q3":
        rho = torch.where(torch.arange(nx, device=dev) < nx // 2, 1.0, 0.5).double()
        rho = rho * torch.from_numpy(1.0 + 1e-3 * rng.standard_normal(nx)).to(dev)
        return rho[None], torch.zeros_like(rho)[None], torch.zeros_like(rho)[None]
    per = cfg["bc"] == "periodic"
    x = (torch.arange(nx, device=dev, dtype=torch.float64) + 0.5) / nx
    y = (torch.arange(ny, device=dev, dtype=torch.float64) + 0.5) / ny
    ux = torch.zeros(ny, nx, device=dev, dtype=torch.float64)
    uy = torch.zeros_like(ux)
    p = torch.zeros_like(ux)
    amp = (cfg["lid_u"] if cfg["lid_u"] else 0.05) / 4
    for _ in range(4):
        kx, ky = (int(k) for k in rng.integers(1, 4, 2))
        a, ph, c = rng.uniform(-1, 1), rng.uniform(0, 2 * math.pi), rng.uniform(-1, 1)
        if per:  # stream function sin(2 pi kx x + ph) sin(2 pi ky y + ph)
            sx, cx = torch.sin(2 * math.pi * kx * x + ph), torch.cos(2 * math.pi * kx * x + ph)
            sy, cy = torch.sin(2 * math.pi * ky * y + ph), torch.cos(2 * math.pi * ky * y + ph)
        else:  # (sin sin)^2: at rest on every wall
            sx, cx = torch.sin(math.pi * kx * x) ** 2, torch.sin(2 * math.pi * kx * x)
            sy, cy = torch.sin(math.pi * ky * y) ** 2, torch.sin(2 * math.pi * ky * y)
        r = kx / ky if kx <= ky else 1.0
        s = ky / kx if ky < kx else 1.0
        ux += a * amp * s * cy[:, None] * sx[None, :]
        uy -= a * amp * r * sy[:, None] * cx[None, :]
        p += c * torch.cos(2 * math.pi * ky * y + ph)[:, None] * torch.cos(2 * math.pi * kx * x)[None, :]
    if cfg["bc"] != "periodic":
        layer = torch.exp(-((1 - y) / 0.05) ** 2)
        taper = torch.ones_like(x) if cfg["bc"] == "channel" else 1 - (2 * x - 1) ** 16
        ux += cfg["lid_u"] * layer[:, None] * taper[None, :]
    return 1.0 + 0.5 * amp * amp * p, ux, uy


def prepare(case, seed):
    if case["kind"] == "batch":
        cfgs = _batch_configs(case)
        dt = torch.float32
        f0 = [_equilibrium(c, *_flow(c, seed + 1000 * k)).to(dt).contiguous() for k, c in enumerate(cfgs)]
        return dict(kind="batch", batch=lbm.Batch(cfgs), f0=f0, steps=case["steps"], dt=dt)
    cfg = _config(case)
    lat = lbm.Lattice(cfg)
    rho, ux, uy = (a.contiguous() for a in _flow(cfg, seed))
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    if case["kind"] == "adjoint":
        f0 = _equilibrium(cfg, rho, ux, uy).to(dt).contiguous()
        return dict(kind="adjoint", lat=lat, f0=f0, T=case["T"], K=case["K"],
                    work=lat.adjoint_work(case["T"], case["K"]))
    if case.get("probe"):
        L = cfg["nx"] - 1
        lat.probe(round(L / 16), round(13 * L / 16), case["steps"])
    return dict(kind="lattice", lat=lat, fields=(rho, ux, uy if cfg["lattice"] == "D2Q9" else None),
                steps=case["steps"], dt=dt, probe=bool(case.get("probe")))


def run(state):
    if state["kind"] == "batch":
        b = state["batch"]
        for k, f in enumerate(state["f0"]):
            b.set_state(k, f)
        b.step(state["steps"])
        return [b.get_state(k, state["dt"]) for k in range(b.n)]
    lat = state["lat"]
    if state["kind"] == "adjoint":
        lat.set_state(state["f0"])
        J, work = lat.adjoint_forward(state["T"], state["K"], state["work"])
        g, gU, gB = lat.adjoint_backward(state["T"], state["K"], work)
        return dict(J=J, df0=g, dU=gU, dbeta=gB)
    lat.init_device(*state["fields"])
    lat.step(state["steps"])
    rho, u = lat.macros(state["dt"])
    out = dict(f=lat.get_state(state["dt"]), rho=rho, u=u)
    if state["probe"]:
        out["signal"] = lat.probe_signal()
    return out


def work(case):
    """Every step reads and writes each population once; the fields that come
    in and the results that go out once."""
    if case["kind"] == "batch":
        cfgs = _batch_configs(case)
        sites = [c["nx"] * c["ny"] for c in cfgs]
        b = BYTES[case["precision"]]
        return dict(bytes=sum(s * (18 * b * case["steps"] + 72) for s in sites),
                    flops=sum(s * FLOPS[c["collision"]] * case["steps"] for s, c in zip(sites, cfgs)))
    q = 3 if case["kind"] == "tube" else 9
    s = case["nx"] * case.get("ny", 1)
    b = BYTES[case["precision"]]
    fl = FLOPS[case["collision"]] * q // 9
    if case["kind"] == "adjoint":
        # forward, recomputation (with its states written), and the adjoint
        # step (state and adjoint read, adjoint written)
        n = case["T"]
        return dict(bytes=s * (q * b * (2 + 3 + 3) * n + 2 * q * b), flops=s * n * (2 * fl + 200))
    out = 8 if case["precision"] == "fp64" else 4
    d = 3 if q == 9 else 2
    return dict(bytes=s * (2 * q * b * case["steps"] + 8 * d + out * (q + d)), flops=s * fl * case["steps"])


# ------------------------------------------------------ the method in 64 bits
CX = {3: [-1, 0, 1], 9: [0, 1, 1, 0, -1, -1, -1, 0, 1]}
CY = {3: [0, 0, 0], 9: [0, 0, -1, -1, -1, 0, 1, 1, 1]}
W = {3: [1 / 6, 2 / 3, 1 / 6], 9: [4 / 9, 1 / 9, 1 / 36, 1 / 9, 1 / 36, 1 / 9, 1 / 36, 1 / 9, 1 / 36]}


def _opp(q, i):
    return 2 - i if q == 3 else (0 if i == 0 else (i + 3) % 8 + 1)


def _q(cfg):
    return 3 if cfg["lattice"] == "D1Q3" else 9


def _vec(v, like):
    return torch.tensor(v, dtype=torch.float64, device=like.device)[:, None, None]


def _equilibrium(cfg, rho, ux, uy):
    q = _q(cfg)
    kind = "entropic" if cfg["collision"] == "elbm" else cfg.get("equilibrium", "poly")
    if q == 9 and kind == "poly_std":
        out = []
        for i in range(9):
            cu = CX[9][i] * ux + CY[9][i] * uy
            out.append(W[9][i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + uy * uy)))
        return torch.stack(out)

    def line(u):
        a = (2 * torch.sqrt(1 + 3 * u * u) - 1) / 6 if kind == "entropic" else (1 + 3 * u * u) / 6
        return [a - u / 2, 1 - 2 * a, a + u / 2]

    px = line(ux)
    if q == 3:
        return torch.stack([rho * p for p in px])
    py = line(uy)
    return torch.stack([rho * px[CX[9][i] + 1] * py[CY[9][i] + 1] for i in range(9)])


def _moments(q, f):
    rho = f.sum(0)
    return rho, (f * _vec(CX[q], f)).sum(0) / rho, (f * _vec(CY[q], f)).sum(0) / rho


def _g(x):
    """(1 + x) ln(1 + x) - x, by its series where the two terms cancel."""
    big = float(x.abs().max()) if x.numel() else 0.0
    n = 6 if big < 1e-3 else 12 if big < 0.03 else 30
    p = torch.full_like(x, (-1) ** n / ((n + 1) * (n + 2)))
    for k in range(n - 1, -1, -1):
        p = p * x + (-1) ** k / ((k + 1) * (k + 2))
    s = x * x * p
    if big < 0.25:
        return s
    xc = x.clamp(min=-1.0)
    return torch.where(x.abs() < 0.25, s, torch.special.xlog1py(1 + xc, xc) - xc)


def _delta_s(f, fe):
    ds = (fe * _g((f - fe) / fe)).sum(0)
    return torch.where(((f < 0) | (fe <= 0)).any(0), torch.full_like(ds, math.inf), ds)


def _alpha(f, fe):
    """The non-trivial root of S(f + alpha (f* - f)) = S(f) above 1 at every
    site (Newton inside a bracket), or alpha_max where there is none."""
    d = (fe - f) / fe
    amax = 1 + 1 / (-d).amax(0).clamp(min=1e-300)
    g0 = (fe * _g(-d)).sum(0)
    def S(a):
        return g0 - (fe * _g((a - 1) * d)).sum(0)
    a = torch.where(amax > 2, torch.full_like(amax, 2.0), 0.5 * (1 + amax))
    lo, hi = torch.ones_like(amax), amax.clone()
    none = (S(amax.clamp(max=1e6)) > 0) & (amax < 1e6) | (f < 0).any(0)
    for _ in range(12):
        s0 = S(a)
        s1 = -(fe * d * torch.log1p(((a - 1) * d).clamp(min=-1 + 1e-15))).sum(0)
        lo, hi = torch.where(s0 > 0, a, lo), torch.where(s0 > 0, hi, a)
        n = a - s0 / s1
        a = torch.where((n > lo) & (n < hi), n, torch.where(torch.isfinite(n) & (n == a), a, 0.5 * (lo + hi)))
    a = torch.where(g0 < 1e-15, torch.full_like(a, 2.0), a)
    return torch.where(none, amax, a)


def _window_median(cfg, ds, fluid):
    """Lower median of Delta S over each site's neighbourhood, clipped to the
    fluid sites."""
    per = {"periodic": (True, True), "channel": (False, True)}.get(cfg["bc"], (False, False))
    vals, cnt = [], torch.zeros_like(ds, dtype=torch.int64)
    ny = ds.shape[0]
    for dy in ((-1, 0, 1) if ny > 1 else (0,)):
        for dx in (-1, 0, 1):
            v, m = torch.roll(ds, (dy, dx), (0, 1)), torch.roll(fluid, (dy, dx), (0, 1)).clone()
            for ax, (dd, p) in enumerate(((dy, per[0]), (dx, per[1]))):
                if dd and not p:
                    m.select(ax, 0 if dd > 0 else -1).fill_(False)
            vals.append(torch.where(m, v, torch.full_like(v, math.inf)))
            cnt += m
    s = torch.stack(vals).sort(0).values
    return s.gather(0, ((cnt - 1).clamp(min=0) // 2)[None])[0]


def _collide(cfg, f, beta, fluid, lag):
    q, coll = _q(cfg), cfg["collision"]
    rho, ux, uy = _moments(q, f)
    fe = _equilibrium(cfg, rho, ux, uy)
    d = f - fe
    if coll == "elbm":
        return f - _alpha(f, fe) * cfg["beta"] * d
    if coll == "mrt" and q == 9:
        M = np.array([[1] * 9, [-4, -1, 2, -1, 2, -1, 2, -1, 2], [4, -2, 1, -2, 1, -2, 1, -2, 1], CX[9],
                      [0, -2, 1, 0, -1, 2, -1, 0, 1], CY[9], [0, 0, -1, 2, -1, 0, 1, -2, 1],
                      [0, 1, 0, -1, 0, 1, 0, -1, 0], [0, 0, -1, 0, 1, 0, -1, 0, 1]], float)
        s = 2 * cfg["beta"]
        rate = np.diag([1, cfg["s_e"], cfg["s_eps"], 1, cfg["s_q"], 1, cfg["s_q"], s, s])
        A = torch.from_numpy(np.linalg.solve(M, rate @ M)).to(f)
        return f - torch.einsum("ij,jyx->iyx", A, d)

    def aggressive():
        r4 = [CX[9][i] ** 2 - CY[9][i] ** 2 for i in range(9)]
        r5 = [CX[9][i] * CY[9][i] for i in range(9)]
        c = (1 - 2 * beta) / 4
        m4, m5 = c * (_vec(r4, f) * d).sum(0), c * (_vec(r5, f) * d).sum(0)
        return fe + _vec(r4, f) * m4 + _vec(r5, f) * m5

    if coll == "mrt2":
        return aggressive()
    F = f - 2 * beta * d
    if coll in ("lbgk", "mrt"):
        return F
    if coll == "positivity":
        neg = F < 0
        lam = torch.where(neg, fe / (fe - F), torch.ones_like(F)).amin(0)
        return fe + lam * (F - fe)
    fd, fed = f.detach(), fe.detach()
    ds = _delta_s(fd, fed)
    if coll in ("ehrenfest", "mrt_limiter"):
        v = torch.where(fluid & (ds > cfg["delta"]), ds, torch.full_like(ds, -1.0)).reshape(-1)
        top = v.topk(min(cfg["topk"], v.numel()))
        sel = torch.zeros_like(v, dtype=torch.bool)
        sel[top.indices[top.values > 0]] = True
        return torch.where(sel.reshape(ds.shape), fe if coll == "ehrenfest" else aggressive(), F)
    if coll == "median":
        med = _window_median(cfg, ds, fluid)
        sel = fluid & (ds > cfg["delta"]) & (med < ds)
        if f.requires_grad:
            # the chosen window site's Delta S depends on f as well: find it
            ds = _delta_s(f, fe)
            med = _window_median(cfg, ds, fluid)
        phi = torch.sqrt(torch.where(sel, med / ds, torch.ones_like(ds)))
        return fe + (1 - 2 * beta) * phi * d
    fin = fluid & torch.isfinite(ds)
    if coll == "threshold":
        v = ds[fin].sort(descending=True).values
        R = cfg["lim_delta0"] * (1 - (2 * cfg["beta"] - 1) ** 2) * float(v.sum())
        cum, n = v.cumsum(0), torch.arange(1, v.numel() + 1, device=v.device)
        over = (cum - n * v >= R).nonzero()  # the first value below the threshold
        k = int(over[0]) if over.numel() else v.numel()
        t = float((cum[k - 1] - R) / k) if k > 0 else float(v[0])
        t = max(t, cfg["delta"])
        phi = torch.where(ds >= t, torch.sqrt(t / ds), torch.ones_like(ds))
    elif coll == "smooth":
        phi = 1 / (1 + cfg["lim_alpha"] * ds ** cfg["lim_k"])
    elif coll == "double_monotonic":
        phi = (1 + (ds / cfg["lim_dst"]) ** cfg["lim_k"]) ** (-0.5 / cfg["lim_k"])
    else:
        now = float(ds[fin].mean())
        E = now if coll == "ensemble" or lag.get("E") is None else lag["E"]
        lag["E"] = now
        y = ds / (cfg["lim_alpha"] * E) if E > 0 else torch.zeros_like(ds)
        phi = (1 + y ** (cfg["lim_k"] - 0.5)) / (1 + y ** cfg["lim_k"]) if E > 0 else torch.ones_like(ds)
    phi = torch.where(torch.isfinite(ds), phi, torch.zeros_like(phi))
    return fe + (1 - 2 * beta) * phi * d


def _diffusive(cfg, f):
    """Section 8's diffusive Maxwell rule at the wall sites (in place)."""
    ny, nx = f.shape[1:]
    one, zero = torch.ones(1, 1, dtype=f.dtype, device=f.device), torch.zeros(1, 1, dtype=f.dtype, device=f.device)
    for ax, at, n, uw in ((1, 0, (0, -1), 0.0), (1, ny - 1, (0, 1), cfg["lid_u"]), (2, 0, (-1, 0), 0.0),
                          (2, nx - 1, (1, 0), 0.0)):
        fe = _equilibrium(cfg, one, zero + uw, zero).reshape(9, 1)
        vn = [CX[9][i] * n[0] + CY[9][i] * n[1] for i in range(9)]
        line = f.select(ax, at)[:, 1:-1]
        gam = sum(line[i] for i in range(9) if vn[i] > 0) / sum(fe[i] for i in range(9) if vn[i] < 0)
        for i in range(9):
            if vn[i] < 0:
                line[i] = gam * fe[i]
    for y in (0, ny - 1):
        for x in (0, nx - 1):
            g = f[:, y, x].clone()
            inside = lambda i: 0 <= x - CX[9][i] < nx and 0 <= y - CY[9][i] < ny  # noqa: E731, B023
            for i in range(9):
                if not inside(i) and inside(_opp(9, i)):
                    f[i, y, x] = g[_opp(9, i)]


def _stream(cfg, F, lid):
    q = _q(cfg)
    px, py = cfg["bc"] in ("periodic", "channel"), cfg["bc"] == "periodic"
    rows = []
    for i in range(q):
        cx, cy, o = CX[q][i], CY[q][i], _opp(q, i)
        g = torch.roll(F[i], (cy, cx), (0, 1))
        if cx and not px:
            k = 0 if cx > 0 else -1
            g[:, k] = F[o][:, k]
        if cy and not py:
            k = 0 if cy > 0 else -1
            g[k] = F[o][k]
            if cy < 0 and cfg["bc"] != "diffusive":
                # a link through the top wall, the corner's own included
                g[k] = F[o][k] - 6 * W[q][o] * CX[q][o] * lid
        rows.append(g)
    return torch.stack(rows)


def _fluid(cfg, like):
    m = torch.ones(like.shape[1:], dtype=torch.bool, device=like.device)
    if cfg["bc"] == "diffusive":
        m[0], m[-1], m[:, 0], m[:, -1] = False, False, False, False
    return m


def _step(cfg, f, beta, lid, fluid, lag):
    if cfg["bc"] == "diffusive":
        f = f.clone()
        _diffusive(cfg, f)
        F = torch.where(fluid, _collide(cfg, f, beta, fluid, lag), f)
    else:
        F = _collide(cfg, f, beta, fluid, lag)
    return _stream(cfg, F, lid)


def _exact_adjoint(case, cfg, f0):
    T, seg = case["T"], 20
    fluid = _fluid(cfg, f0)
    ck, f = [], f0
    with torch.no_grad():
        for t in range(T):
            if t % seg == 0:
                ck.append(f)
            f = _step(cfg, f, cfg["beta"], cfg["lid_u"], fluid, {})

    def energy(f):
        rho, ux, uy = _moments(9, f)
        return 0.5 * (rho * (ux * ux + uy * uy)).sum()

    f = f.requires_grad_(True)
    J = energy(f)
    (lam,) = torch.autograd.grad(J, f)
    gU = gB = 0.0
    for s in range(len(ck) - 1, -1, -1):
        f = ck.pop().detach().requires_grad_(True)
        b = torch.tensor(cfg["beta"], dtype=torch.float64, device=f.device, requires_grad=True)
        u = torch.tensor(cfg["lid_u"], dtype=torch.float64, device=f.device, requires_grad=True)
        h = f
        for _ in range(min(seg, T - s * seg)):
            h = _step(cfg, h, b, u, fluid, {})
        lam, du, db = torch.autograd.grad(h, (f, u, b), lam)
        gU, gB = gU + float(du), gB + float(db)
    return dict(J=float(J), df0=lam, dU=gU, dbeta=gB)


def exact(case, seed):
    if case["kind"] == "batch":
        out = []
        for k, cfg in enumerate(_batch_configs(case)):
            f = _equilibrium(cfg, *_flow(cfg, seed + 1000 * k)).float().double()
            fluid = _fluid(cfg, f)
            for _ in range(case["steps"]):
                f = _step(cfg, f, cfg["beta"], cfg["lid_u"], fluid, {})
            out.append(f)
        return out
    cfg = _config(case)
    cfg.setdefault("beta", 1.0 / (6.0 * cfg["nu"] + 1.0))
    cfg.setdefault("equilibrium", "poly")
    f = _equilibrium(cfg, *_flow(cfg, seed))
    fluid = _fluid(cfg, f)
    if case["kind"] == "adjoint":
        # through the median filter the gradient is left to the forward value
        f = f.float().double()
        if case["collision"] == "median":
            with torch.no_grad():
                for _ in range(case["T"]):
                    f = _step(cfg, f, cfg["beta"], cfg["lid_u"], fluid, {})
                rho, ux, uy = _moments(9, f)
            return dict(J=float(0.5 * (rho * (ux * ux + uy * uy)).sum()), df0=None, dU=None, dbeta=None)
        return _exact_adjoint(case, cfg, f)
    lag, sig = {}, []
    L = cfg["nx"] - 1
    at = (slice(None), round(13 * L / 16), round(L / 16))
    for _ in range(case["steps"]):
        f = _step(cfg, f, cfg["beta"], cfg["lid_u"], fluid, lag)
        if case.get("probe"):
            sig.append(torch.stack([m.squeeze() for m in _moments(9, f[at][:, None, None])[1:]]))
    rho, ux, uy = _moments(_q(cfg), f)
    out = dict(f=f, rho=rho, u=torch.stack([ux, uy]) if _q(cfg) == 9 else ux[None])
    if case.get("probe"):
        out["signal"] = torch.stack(sig)
    return out
