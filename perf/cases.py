"""The work that a user of this library has it do, as cases that can be measured.

A case is a dict of plain values; `prepare` makes its problem on the GPU from
a seed, `run` takes it once through the public calls of
paper_2507_03975_gb300.gsis, `work` says what one pass cannot do without and
`exact` restates the result in plain torch, in 64 bits.

Kinds: "sweep" (gsis.transport_sweep), "synthetic" (gsis.synthetic_step),
"solve" (gsis.solve: GSIS or source iteration, first or second order upwind),
"batch" (gsis.solve_batch), "td" (gsis.td_solve), "adjoint"
(gsis.solve_differentiable and its backward pass), "td_adjoint"
(gsis.td_adjoint).

Media: "uniform" (sigma_t near 10, ratio 0.99, q near 1, vacuum), "random"
(per-cell sigma_t over three decades, non-uniform mesh, inflow on every
wall), "field" (a smooth field over six decades, q = 1, vacuum) and
"channel" (bulk 2000, bent channel 0.2, unit intensity through the left wall).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2507_03975_gb300 import gsis

FOUR_PI = 4.0 * math.pi


def listed():
    return [
        # the smallest call: one kinetic step of the 64x64 S8 problem (set-up and launches count)
        dict(name="sweep_64_S8", kind="sweep", nx=64, ny=64, order=8, medium="uniform", fp32=False),
        # an ordinary kinetic step, as a program with its own iteration calls it
        dict(name="sweep_256_S12", kind="sweep", nx=256, ny=256, order=12, medium="channel", fp32=False),
        # FP32 intensities on an odd, non-uniform mesh with inflow on every wall
        dict(name="sweep_641x470_S6_f32", kind="sweep", nx=641, ny=470, order=6, medium="random", fp32=True),
        # the synthetic step alone, solved to its default tolerance, a mesh of odd sides beyond one cluster
        dict(name="synthetic_513x290", kind="synthetic", nx=513, ny=290, medium="random"),
        # a small steady problem with every option at its default
        dict(name="gsis_64_S8", kind="solve", scheme="gsis", nx=64, ny=64, order=8, medium="uniform", fp32=False,
             beta=0.0, tol=1e-8, synth_max_iter=20000, spatial_order=1, limiter=0, max_iter=2000, iters=29),
        # the same problem by source iteration, the method the scheme is compared with
        dict(name="si_64_S8", kind="solve", scheme="si", nx=64, ny=64, order=8, medium="uniform", fp32=False,
             beta=0.0, tol=1e-8, synth_max_iter=20000, spatial_order=1, limiter=0, max_iter=2000, iters=252),
        # the steady multiscale channel at the benchmark's settings
        dict(name="gsis_channel_256_S12", kind="solve", scheme="gsis", nx=256, ny=256, order=12, medium="channel",
             fp32=False, beta=10.0, tol=1e-8, synth_max_iter=2, spatial_order=1, limiter=0, max_iter=2000, iters=103),
        # second-order upwind with the limiter to the criterion of the paper's steady tests
        dict(name="uw2_channel_256_S12", kind="solve", scheme="gsis", nx=256, ny=256, order=12, medium="channel",
             fp32=False, beta=10.0, tol=1e-6, synth_max_iter=2, spatial_order=2, limiter=0, max_iter=250, iters=204),
        # many uneven problems at once, FP32 intensities (throughput use)
        dict(name="batch_24_f32", kind="batch", count=24, side_lo=32, side_hi=256, fp32=True, tol=1e-6,
             synth_max_iter=2, max_iter=400, iters=62),
        # the largest: the first steps of the 1024x1024 S16 radiation-material run, FP64
        dict(name="td_1024_S16", kind="td", n=1024, order=16, nsteps=8, fp32=False, tol=1e-8, synth_max_iter=6,
             predictor=2, iters=70),
        # the FP32 form of such a run on a quarter of the mesh
        dict(name="td_512_S12_f32", kind="td", n=512, order=12, nsteps=12, fp32=True, tol=1e-7, synth_max_iter=6,
             predictor=2, iters=90),
        # gradient of a time-dependent run with checkpoints (forward, recomputation and transposed sweeps)
        dict(name="td_adjoint_200_S8", kind="td_adjoint", n=200, order=8, nsteps=6, fp32=False, tol=1e-8,
             synth_max_iter=50, predictor=2, iters=60),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["sweep", "sweep", "sweep", "synthetic", "solve", "solve", "solve", "batch", "td", "td",
                       "adjoint", "td_adjoint"])
    order = rng.choice([4, 6, 8, 10, 12, 14, 16])
    fp32 = rng.random() < 0.4
    if kind == "sweep":
        return dict(kind=kind, nx=_log_int(rng, 24, 1000), ny=_log_int(rng, 24, 1000), order=order,
                    medium=rng.choice(["uniform", "random", "channel"]), fp32=fp32)
    if kind == "synthetic":
        return dict(kind=kind, nx=_log_int(rng, 24, 900), ny=_log_int(rng, 24, 900),
                    medium=rng.choice(["uniform", "random"]))
    if kind == "solve":
        scheme = rng.choice(["gsis", "gsis", "si"])
        medium = "uniform" if scheme == "si" else rng.choice(["uniform", "field", "channel"])
        so = 2 if scheme == "gsis" and rng.random() < 0.25 else 1
        n = _log_int(rng, 24, 280)
        # source iteration and second-order runs are stopped after a fixed effort, as a comparison run is
        return dict(kind=kind, scheme=scheme, nx=n, ny=n if medium == "channel" else _log_int(rng, 24, 280),
                    order=order, medium=medium, fp32=fp32, beta=0.0 if medium == "uniform" else 10.0,
                    tol=1e-6 if fp32 else 1e-8, synth_max_iter=20000 if medium == "uniform" else 2,
                    spatial_order=so, limiter=rng.choice([0, 1]), max_iter=60 if so == 2 or scheme == "si" else 300,
                    iters=60)
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(3, 24), side_lo=32, side_hi=_log_int(rng, 48, 256), fp32=fp32,
                    tol=1e-6, synth_max_iter=2, max_iter=300, iters=60)
    if kind == "td":
        return dict(kind=kind, n=_log_int(rng, 64, 900), order=order, nsteps=rng.randint(1, 6), fp32=fp32,
                    tol=1e-7 if fp32 else 1e-8, synth_max_iter=6, predictor=rng.choice([0, 1, 2]), iters=60)
    if kind == "adjoint":
        return dict(kind=kind, nx=_log_int(rng, 24, 160), ny=_log_int(rng, 24, 160), order=order, medium="uniform",
                    fp32=False, tol=1e-8, max_iter=300, iters=60)
    return dict(kind=kind, n=_log_int(rng, 32, 200), order=rng.choice([4, 6, 8]), nsteps=rng.randint(2, 6),
                fp32=False, tol=1e-8, synth_max_iter=50, predictor=rng.choice([0, 2]), iters=60)


# ------------------------------------------------------------------ inputs
_MU1 = {4: math.sqrt((4.0 - math.sqrt(6.4)) / 12.0), 6: 0.2666355, 8: 0.2182179, 10: 0.1893213, 12: 0.1672126,
        14: 0.1519859, 16: 0.1389568}


def _df(k):
    return math.prod(range(k, 0, -2)) if k > 1 else 1


def quadrature(order):
    """Level-symmetric S_order set of the 2D problem: (mu, eta, w), sum w = 4 pi,
    K = order (order + 2) / 2, quadrants (+,+), (-,+), (+,-), (-,-)."""
    n, m1 = order // 2, _MU1[order]
    lev = np.sqrt(m1 * m1 + 2.0 * (1.0 - 3.0 * m1 * m1) / (order - 2) * np.arange(n))
    abc = [(a, b, n - 1 - a - b) for a in range(n) for b in range(n - a)]
    cls = [tuple(sorted(t)) for t in abc]
    names = sorted(set(cls))
    ci = np.array([names.index(c) for c in cls])
    p = lev[np.array(abc)]
    rows, rhs = [], []
    for a, b, c in ((a, b, c) for a in range(n) for b in range(n - a) for c in range(n - a - b)):
        row = np.zeros(len(names))
        np.add.at(row, ci, p[:, 0] ** (2 * a) * p[:, 1] ** (2 * b) * p[:, 2] ** (2 * c))
        rows.append(row)
        rhs.append(_df(2 * a - 1) * _df(2 * b - 1) * _df(2 * c - 1) / _df(2 * (a + b + c) + 1))
    w = np.linalg.lstsq(np.array(rows), np.array(rhs), rcond=None)[0][ci] * math.pi
    w *= math.pi / w.sum()
    sx, sy = (1, -1, 1, -1), (1, 1, -1, -1)
    return (np.concatenate([s * p[:, 0] for s in sx]), np.concatenate([s * p[:, 1] for s in sy]),
            np.concatenate([w] * 4))


def _channel_mask(nx, ny, rng):
    """[ny, nx] mask of a bent channel on a 256 x 256 base grid, sampled to the mesh."""
    m = np.zeros((256, 256), dtype=bool)
    x, y = 0, int(rng.integers(64, 193))
    while x < 256:
        x1 = min(255, x + int(rng.integers(32, 97)))
        m[max(0, y - 4):y + 4, x:x1 + 1] = True
        x = x1
        if x >= 255:
            break
        y1 = int(np.clip(y + int(rng.integers(8, 33)) * (1 if rng.random() < 0.5 else -1), 8, 240))
        m[max(0, min(y, y1) - 4):max(y, y1) + 4, max(0, x - 4):x + 4] = True
        y = y1
    return m[np.ix_(np.arange(ny) * 256 // ny, np.arange(nx) * 256 // nx)]


def _smooth_field(nx, ny, rng):
    ks = [(a, b) for a in range(-4, 5) for b in range(-4, 5) if 0 < a * a + b * b <= 16]
    X, Y = (np.arange(nx) + 0.5) / nx, ((np.arange(ny) + 0.5) / ny)[:, None]
    g = np.zeros((ny, nx))
    for t in rng.choice(len(ks), 16, replace=False):
        g += np.cos(2.0 * math.pi * (ks[t][0] * X + ks[t][1] * Y) + rng.uniform(0.0, 2.0 * math.pi))
    return torch.erf(torch.from_numpy(g * math.sqrt(2.0 / 16) / math.sqrt(2.0))).numpy()


def _problem(nx, ny, order, medium, rng):
    """Host arrays of one problem (mesh, quadrature) and its device arrays."""
    mu, eta, w = quadrature(order)
    N, K = nx * ny, len(mu)
    dx, dy = np.full(nx, 1.0 / nx), np.full(ny, 1.0 / ny)
    inflow, q = None, np.ones(N)
    if medium == "uniform":
        st, ratio, q = 10.0 * rng.uniform(0.95, 1.05, N), 0.99, rng.uniform(0.9, 1.1, N)
    elif medium == "random":
        dx, dy = rng.uniform(0.5, 1.5, nx), rng.uniform(0.5, 1.5, ny)
        dx, dy = dx / dx.sum(), dy / dy.sum()
        st, ratio, q = 10.0 ** rng.uniform(-1.0, 2.0, N), rng.uniform(0.3, 0.99, N), rng.uniform(0.0, 2.0, N)
        inflow = rng.uniform(0.0, 1.0, (2 * (nx + ny), K))
    elif medium == "field":
        st = 10.0 ** (-2.0 + 3.0 * (1.0 + _smooth_field(nx, ny, rng).reshape(-1)))
        ratio = rng.uniform(0.5, 0.9999)
    else:
        st = np.where(_channel_mask(nx, ny, rng).reshape(-1), 0.2, 2000.0) * rng.uniform(0.99, 1.01)
        ratio, q = 0.999, np.zeros(N)
        inflow = np.zeros((2 * (nx + ny), K))
        inflow[:ny] = 1.0
    t = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).cuda()  # noqa: E731
    return dict(nx=nx, ny=ny, dx=dx, dy=dy, mu=mu, eta=eta, w=w, sigma_a=t(st - ratio * st), sigma_s=t(ratio * st),
                q=t(q), inflow=t(inflow))


def _inputs(case, seed):
    """The problem of a case, with what the call takes beyond it."""
    rng = np.random.Generator(np.random.PCG64(seed))
    kind = case["kind"]
    if kind == "batch":
        lo, hi = case["side_lo"], case["side_hi"]
        sides = [int(round(lo * (hi / lo) ** ((i + 0.5) / case["count"]))) for i in range(case["count"])]
        return [_problem(s, s, (8, 10, 12, 14, 16)[i % 5], "field", rng) for i, s in enumerate(sides)]
    nx, ny = (case["n"], case["n"]) if kind in ("td", "td_adjoint") else (case["nx"], case["ny"])
    p = _problem(nx, ny, case.get("order", 4), case.get("medium", "channel"), rng)
    N, dev = nx * ny, p["sigma_a"].device
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    u = lambda n, lo, hi: torch.empty(n, dtype=torch.float64, device=dev).uniform_(lo, hi, generator=g)  # noqa: E731
    if kind == "sweep":
        p["rho"] = u(N, 0.5, 1.5)
    elif kind == "synthetic":
        p.update(rho_half=u(N, 0.5, 1.5), F_half=u(2 * N, -0.1, 0.1), bflux=u(2 * (nx + ny), 0.0, 0.3))
    elif kind == "adjoint":
        p["g"] = u(N, 0.0, 1.0)
    elif kind in ("td", "td_adjoint"):
        p["T0"] = u(N, 0.1, 0.11)
        p["rho0"] = p["T0"] ** 4
        if kind == "td_adjoint":
            p.update(g_rho=u(N, 0.0, 1.0), g_T=u(N, 0.0, 1.0))
    return p


def _options(case):
    kind = case["kind"]
    o = dict(precision=gsis.FP32_SWEEP if case.get("fp32") else gsis.FP64)
    for k in ("tol", "max_iter", "synth_max_iter", "beta", "spatial_order", "limiter"):
        if k in case:
            o[k] = case[k]
    if kind == "solve":
        o["scheme"] = gsis.SCHEME_SI if case["scheme"] == "si" else gsis.SCHEME_GSIS
        if case["spatial_order"] == 2 or case["max_iter"] <= 60:
            o["check_every"] = 8
    if kind == "batch":
        o["beta"] = 10.0
    if kind == "td":
        o.update(check_every=5, max_iter=400)
        if case["fp32"]:
            o.update(check_every=2, stall_window=5)
    return gsis.default_options(**o)


def prepare(case, seed):
    kind, opt = case["kind"], _options(case)
    p = _inputs(case, seed)
    s = dict(kind=kind, p=p, opt=opt, case=case)
    if kind == "batch":
        n = gsis.batch_workspace_bytes(p, opt)
    else:
        s["host"] = h = (p["dx"], p["dy"], p["mu"], p["eta"], p["w"])
        if kind == "td":
            n = gsis.td_workspace_bytes(*h, opt)
        elif kind == "td_adjoint":
            n = gsis.td_adjoint_workspace_bytes(*h, 1e-3, case["nsteps"], 3, options=opt)
        elif kind == "synthetic":
            n = gsis.workspace_bytes(*h[:2], options=opt)
        elif kind == "adjoint":
            n = 0   # the autograd function takes its own
            p["sigma_a"].requires_grad_(True)
            p["sigma_s"].requires_grad_(True)
        else:
            n = gsis.workspace_bytes(*h, opt)
    s["ws"] = torch.empty(max(n, 1), dtype=torch.uint8, device="cuda")   # kept by the caller between calls
    return s


def run(s):
    kind, p, opt, ws, case = s["kind"], s["p"], s["opt"], s["ws"], s["case"]
    if kind == "batch":
        r = gsis.solve_batch(p, opt, workspace=ws)["results"]
        return [(x["rho"], x["F"]) for x in r]
    mat = (p["sigma_a"], p["sigma_s"], p["q"])
    if kind == "sweep":
        r = gsis.transport_sweep(*s["host"], *mat, p["rho"], inflow=p["inflow"], options=opt, workspace=ws)
        return r["rho"], r["F"], r["P"], r["bflux"]
    if kind == "synthetic":
        r = gsis.synthetic_step(p["dx"], p["dy"], *mat, p["rho_half"], p["F_half"], p["bflux"], options=opt, workspace=ws)
        return r["rho"], r["hot"], r["rhs"]
    if kind == "solve":
        r = gsis.solve(*s["host"], *mat, inflow=p["inflow"], options=opt, workspace=ws)
        return r["rho"], r["F"], r["P"]
    if kind == "td":
        r = gsis.td_solve(*s["host"], *mat, p["rho0"], p["T0"], 1e-3, case["nsteps"], inflow=p["inflow"], options=opt,
                          workspace=ws, predictor=case["predictor"])
        return r["rho"], r["T"], r["F"]
    if kind == "adjoint":
        rho = gsis.solve_differentiable(*s["host"], *mat, inflow=p["inflow"], options=opt)
        ga, gs = torch.autograd.grad(rho, mat[:2], p["g"])
        return rho.detach(), ga, gs
    r = gsis.td_adjoint(*s["host"], *mat, p["rho0"], p["T0"], 1e-3, case["nsteps"], dJ_drho=p["g_rho"], dJ_dT=p["g_T"],
                        checkpoint_every=3, inflow=p["inflow"], options=opt, workspace=ws,
                        predictor=case["predictor"])
    return r["rho"], r["T"], r["grad_sigma_a"], r["grad_sigma_s"], r["grad_rho0"], r["grad_T0"]


def work(case):
    """Bytes: the caller's arrays once.  Operations: per update (cell x direction) of each of the iterations
    that such a case takes (`iters`) five in the sweep and five in two moments of a pair of updates."""
    kind = case["kind"]
    K = lambda order: order * (order + 2) // 2  # noqa: E731
    if kind == "batch":
        lo, hi, c = case["side_lo"], case["side_hi"], case["count"]
        N = [int(round(lo * (hi / lo) ** ((i + 0.5) / c))) ** 2 for i in range(c)]
        u = sum(n * K((8, 10, 12, 14, 16)[i % 5]) for i, n in enumerate(N))
        return {"bytes": 48.0 * sum(N), "flops": 9.0 * u * case["iters"]}
    nx, ny = (case["n"], case["n"]) if kind in ("td", "td_adjoint") else (case["nx"], case["ny"])
    N, k = nx * ny, K(case.get("order", 4))
    if kind == "synthetic":   # a solve of a five-point system: a few tens of operations per cell and digit
        return {"bytes": 8.0 * N * 10, "flops": 20.0 * 12 * N}
    inflow = 16.0 * (nx + ny) * k if case.get("medium", "channel") != "uniform" else 0.0
    arrays = {"sweep": 10, "solve": 9, "td": 9, "adjoint": 7, "td_adjoint": 13}[kind]
    return {"bytes": 8.0 * N * arrays + inflow, "flops": 9.0 * N * k * case.get("iters", 1)}


# ---------------------------------------------------------- the same, in plain torch
def _sweep(p, src):
    """First-order-upwind sweep of every ordinate by anti-diagonals; the moments and the boundary flux."""
    nx, ny, dev = p["nx"], p["ny"], src.device
    f64 = lambda a: torch.as_tensor(np.asarray(a), dtype=torch.float64, device=dev)  # noqa: E731
    K4 = len(p["mu"]) // 4
    mu, eta, w = (f64(p[n]).view(4, K4) for n in ("mu", "eta", "w"))
    dx, dy = f64(p["dx"]), f64(p["dy"])
    st = (p["sigma_a"] + p["sigma_s"]).detach().view(ny, nx)
    flips = [[], [1], [0], [0, 1]]
    S = torch.stack([torch.flip(src.view(ny, nx), f) for f in flips])
    ST = torch.stack([torch.flip(st, f) for f in flips])
    DX = torch.stack([torch.flip(dx, [0]) if 1 in f else dx for f in flips])
    DY = torch.stack([torch.flip(dy, [0]) if 0 in f else dy for f in flips])
    inW = torch.zeros(4, K4, ny, dtype=torch.float64, device=dev)
    inS = torch.zeros(4, K4, nx, dtype=torch.float64, device=dev)
    if p["inflow"] is not None:
        inf = p["inflow"].view(2 * (nx + ny), 4, K4)
        for i, f in enumerate(flips):
            a = inf[ny:2 * ny, i] if 1 in f else inf[:ny, i]
            b = inf[2 * ny + nx:, i] if 0 in f else inf[2 * ny:2 * ny + nx, i]
            inW[i] = torch.flip(a, [0]).T if 0 in f else a.T
            inS[i] = torch.flip(b, [0]).T if 1 in f else b.T
    M = torch.stack([w, w * mu, w * eta, w * mu * mu, w * mu * eta, w * eta * eta], 1)   # [4, 6, K4]
    out = torch.zeros(4, 6, ny, nx, dtype=torch.float64, device=dev)
    east = torch.zeros(4, K4, ny, dtype=torch.float64, device=dev)
    north = torch.zeros(4, K4, nx, dtype=torch.float64, device=dev)
    prev = torch.zeros(4, K4, ny, dtype=torch.float64, device=dev)
    am, ae = mu.abs()[..., None], eta.abs()[..., None]
    for t in range(nx + ny - 1):
        j0, j1 = max(0, t - nx + 1), min(ny - 1, t)
        j = torch.arange(j0, j1 + 1, device=dev)
        i = t - j
        W, So = prev[..., j0:j1 + 1].clone(), torch.zeros(4, K4, j1 - j0 + 1, dtype=torch.float64, device=dev)
        if j0 > 0:
            So[:] = prev[..., j0 - 1:j1]
        elif j1 > 0:
            So[..., 1:] = prev[..., :j1]
        if j0 == 0:
            So[..., 0] = inS[..., t]
        if t <= ny - 1:
            W[..., -1] = inW[..., t]
        a, b = am / DX[:, None, i], ae / DY[:, None, j]
        cur = (S[:, j, i][:, None] + a * W + b * So) / (ST[:, j, i][:, None] + a + b)
        out[:, :, j, i] = torch.matmul(M, cur)
        if t >= nx - 1:
            east[..., j0] = cur[..., 0]
        if t >= ny - 1:
            north[..., t - ny + 1] = cur[..., -1]
        prev[..., j0:j1 + 1] = cur
    m = sum(torch.flip(out[i], [d + 1 for d in f]) for i, f in enumerate(flips)).reshape(6, -1)
    fb = torch.zeros(2 * (nx + ny), dtype=torch.float64, device=dev)
    wm, we = (w * mu)[..., None], (w * eta)[..., None]
    for i, f in enumerate(flips):
        o, n = (wm[i] * east[i]).sum(0), (wm[i] * inW[i]).sum(0)
        e, v = (we[i] * north[i]).sum(0), (we[i] * inS[i]).sum(0)
        if 0 in f:
            o, n = torch.flip(o, [0]), torch.flip(n, [0])
        if 1 in f:
            e, v = torch.flip(e, [0]), torch.flip(v, [0])
        out_w, out_s = 1 in f, 0 in f   # the walls that the ordinates of this quadrant leave through
        fb[:ny] += -o if out_w else -n
        fb[ny:2 * ny] += n if out_w else o
        fb[2 * ny:2 * ny + nx] += -e if out_s else -v
        fb[2 * ny + nx:] += v if out_s else e
    return m, fb


def _synthetic(p, rho_h, F, fb, guess):
    """The synthetic step: high-order terms, right-hand side and the solution (CG with a
    diagonal preconditioner, restarted on the true residual); (rho, hot, rhs)."""
    nx, ny, dev = p["nx"], p["ny"], rho_h.device
    dx = torch.as_tensor(p["dx"], device=dev)[None, :]
    dy = torch.as_tensor(p["dy"], device=dev)[:, None]
    v = lambda a: a.detach().view(ny, nx)  # noqa: E731
    sa, st, r = v(p["sigma_a"]), v(p["sigma_a"] + p["sigma_s"]), v(rho_h)

    def grad(h, axis):
        """Adaptive least squares along one axis: neighbours at their optically scaled distance."""
        h = h.expand(ny, nx)
        n = st.shape[axis]
        a, b = [st.narrow(axis, k, n - 1) for k in (0, 1)]
        ha, hb = [h.narrow(axis, k, n - 1) for k in (0, 1)]
        up, dn = 0.5 * (ha + b / a * hb), -0.5 * (hb + a / b * ha)
        dr = r.narrow(axis, 1, n - 1) - r.narrow(axis, 0, n - 1)
        num, den = torch.zeros_like(r), torch.zeros_like(r)
        num.narrow(axis, 0, n - 1).add_(up * dr)
        den.narrow(axis, 0, n - 1).add_(up * up)
        num.narrow(axis, 1, n - 1).add_(-dn * dr)
        den.narrow(axis, 1, n - 1).add_(dn * dn)
        return torch.where(den > 0, num / den.clamp_min(1e-300), torch.zeros_like(num))

    hx = v(F[:nx * ny]) + grad(dx, 1) / (3.0 * st)
    hy = v(F[nx * ny:]) + grad(dy, 0) / (3.0 * st)
    ox, oy = st * dx, st * dy
    cx = dy * 2.0 / (3.0 * (ox[:, :-1] + ox[:, 1:]))
    cy = dx * 2.0 / (3.0 * (oy[:-1] + oy[1:]))
    bx, by = dy * (2.0 / (3.0 * ox) + 0.25), dx * (2.0 / (3.0 * oy) + 0.25)
    diag = dx * dy * sa
    b = dx * dy * v(p["q"])
    diag[:, :-1] += cx
    diag[:, 1:] += cx
    diag[:-1] += cy
    diag[1:] += cy
    fx, fy = 0.5 * dy * (hx[:, :-1] + hx[:, 1:]), 0.5 * dx * (hy[:-1] + hy[1:])
    b[:, :-1] -= fx
    b[:, 1:] += fx
    b[:-1] -= fy
    b[1:] += fy
    for sl, be, h, f in ((np.s_[:, 0], bx, dy[:, 0], fb[:ny]), (np.s_[:, -1], bx, dy[:, 0], fb[ny:2 * ny]),
                         (np.s_[0], by, dx[0], fb[2 * ny:2 * ny + nx]), (np.s_[-1], by, dx[0], fb[2 * ny + nx:])):
        diag[sl] += be[sl]
        b[sl] += be[sl] * r[sl] - h * f

    def D(x):
        y = diag * x
        y[:, :-1] -= cx * x[:, 1:]
        y[:, 1:] -= cx * x[:, :-1]
        y[:-1] -= cy * x[1:]
        y[1:] -= cy * x[:-1]
        return y

    x = v(guess).clone()
    for _ in range(3):
        res = b - D(x)
        z = res / diag
        d, rz = z.clone(), (res * z).sum()
        e, stop = torch.zeros_like(x), 1e-30 * float((b * b / diag).sum())
        for k in range(12000):
            q = D(d)
            al = rz / (d * q).sum()
            e += al * d
            res = res - al * q
            z = res / diag
            new = (res * z).sum()
            if k % 50 == 49 and not float(new) > stop:
                break
            d = z + (new / rz) * d
            rz = new
        x = x + torch.nan_to_num(e)
    return x.reshape(-1), torch.cat([hx.reshape(-1), hy.reshape(-1)]), b.reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        p = _inputs(case, seed)
        m, fb = _sweep(p, (p["sigma_s"] * p["rho"] + p["q"]) / FOUR_PI)
        return m[0], m[1:3].reshape(-1), m[3:].reshape(-1), fb
    if kind == "synthetic":
        p = _inputs(case, seed)
        return _synthetic(p, p["rho_half"], p["F_half"], p["bflux"], p["rho_half"])
    # whole solves: where the iteration is the plain one, solved exactly, and small
    if kind != "solve" or case["beta"] > 0 or case["spatial_order"] != 1 or case["fp32"]:
        return None
    if (case["nx"] + case["ny"]) * case["iters"] > 40000 or case["scheme"] == "gsis" and case["nx"] * case["ny"] > 10000:
        return None
    p = _inputs(case, seed)
    V = (torch.as_tensor(p["dx"])[None, :] * torch.as_tensor(p["dy"])[:, None]).reshape(-1).cuda()
    rho = torch.zeros(case["nx"] * case["ny"], dtype=torch.float64, device="cuda")
    for _ in range(case["max_iter"]):
        m, fb = _sweep(p, (p["sigma_s"] * rho + p["q"]) / FOUR_PI)
        new = m[0] if case["scheme"] == "si" else _synthetic(p, m[0], m[1:3].reshape(-1), fb, rho)[0]
        err = math.sqrt(float(((new - rho) ** 2 * V).sum() / (new ** 2 * V).sum()))
        rho = new
        if err < case["tol"]:
            break
    P = m[3:].clone()
    if case["scheme"] == "gsis":
        P[0] += (rho - m[0]) / 3.0
        P[2] += (rho - m[0]) / 3.0
    return rho, m[1:3].reshape(-1), P.reshape(-1)
