"""The performance cases: what programs have this solver do, through its
public entry points, over the range of grids and options that it serves.

Kinds of case:
  solve     a time step's elliptic problem: the seven coefficient fields of
            Eq. 10 are handed over and L(Phi) = R is solved from a zero guess
  ensemble  independent problems of several grid sizes in one launch
  apply     L and the preconditioner on their own, as a program with a Krylov
            method of its own calls them at each of its iterations
  step      time steps of the semi-implicit shallow-water model
  net       the learned preconditioner applied to one residual
  grad      the network's loss and parameter gradients over a batch
  train     AdamW steps of the network, and its parameters afterwards

Inputs are smooth seeded states on the sphere (sums of plane waves in the
unit vector, so they are smooth across the poles too), with depths of 8000 m
within 5 %, winds up to 40 m/s and a polar absorber: the sizes the solver
meets in the model.
"""
import math

import numpy as np
import torch

import paper_2103_16120_gb300 as sw

A_EARTH, OMEGA, GRAV = 6.371e6, 7.292e-5, 9.80616
PREC = {"fp64": sw.SW_PREC_FP64, "fp16": sw.SW_PREC_MIXED_FP16, "bf16": sw.SW_PREC_MIXED_BF16}


def listed():
    return [
        # the smallest grid of the paper in full precision: latency and launches
        {"name": "solve fp64 128x64", "kind": "solve", "prec": "fp64", "nx": 128, "ny": 64},
        # the paper's finest grid, mixed precision: the usual model resolution
        {"name": "solve fp16 512x256", "kind": "solve", "prec": "fp16", "nx": 512, "ny": 256},
        # the largest grid of the benchmark, mixed precision
        {"name": "solve fp16 2048x1024", "kind": "solve", "prec": "fp16", "nx": 2048, "ny": 1024},
        # a one-degree grid with a row on the equator: neither size a power of two
        {"name": "solve bf16 360x181", "kind": "solve", "prec": "bf16", "nx": 360, "ny": 181},
        # a large grid in full precision: reference solutions and training data
        {"name": "solve fp64 1024x512", "kind": "solve", "prec": "fp64", "nx": 1024, "ny": 512},
        # an ensemble forecast on the paper's three grids
        {"name": "ensemble fp16 64", "kind": "ensemble", "prec": "fp16", "nx": 128, "ny": 64, "n0": 32, "n1": 24, "n2": 8},
        # a Krylov method of the caller's own, full precision, the largest grid
        {"name": "apply fp64 2048x1024", "kind": "apply", "prec": "fp64", "nx": 2048, "ny": 1024},
        # the same in mixed precision on a quarter-degree grid (no power of two)
        {"name": "apply fp16 1440x721", "kind": "apply", "prec": "fp16", "nx": 1440, "ny": 721},
        # the model itself: two time steps from a state without history
        {"name": "step fp16 512x256", "kind": "step", "prec": "fp16", "nx": 512, "ny": 256, "steps": 2},
        # the learned preconditioner on one residual: inference at batch 1
        {"name": "net 512x256", "kind": "net", "nx": 512, "ny": 256},
        # a small batch on the smallest grid: gradients for an optimiser of the caller's own
        {"name": "grad 8 x 128x64", "kind": "grad", "batch": 8, "nx": 128, "ny": 64},
        # training at the size the network is trained on
        {"name": "train 32 x 256x128", "kind": "train", "batch": 32, "nx": 256, "ny": 128, "steps": 2},
    ]


def _spread(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid(rng, hi, lo=64):
    """nx even (half the time a power of two), ny about nx / 2, odd at times."""
    nx = 2 * round(_spread(rng, lo, hi) / 2)
    if rng.random() < 0.5:
        nx = 1 << max(6, int(math.log2(nx)))
    return nx, nx // 2 + rng.choice((0, 0, 1, -1))


def draw(rng):
    kind = rng.choice(("solve", "solve", "solve", "ensemble", "apply", "apply", "step", "net", "grad", "train"))
    prec = rng.choice(("fp64", "fp16", "bf16"))
    if kind == "solve":
        nx, ny = _grid(rng, 1024 if prec == "fp64" else 1440)
        return {"kind": kind, "prec": prec, "nx": nx, "ny": ny}
    if kind == "ensemble":
        nx, ny = _grid(rng, 192)
        return {"kind": kind, "prec": prec, "nx": nx, "ny": ny, "n0": rng.randint(1, 32), "n1": rng.randint(0, 16),
                "n2": rng.randint(0, 4)}
    if kind == "apply":
        nx, ny = _grid(rng, 2049)
        return {"kind": kind, "prec": prec, "nx": nx, "ny": ny}
    if kind == "step":
        nx, ny = _grid(rng, 768)
        return {"kind": kind, "prec": prec, "nx": nx, "ny": ny, "steps": rng.randint(1, 3)}
    nx = rng.choice((64, 128, 256, 512, 768, 1024)) if kind == "net" else rng.choice((64, 128, 256, 512))
    ny = max(8, 4 * round(nx / 8 + rng.choice((0, 0, -1, 1, 2))))
    if kind == "net":
        return {"kind": kind, "nx": nx, "ny": ny}
    batch = max(1, min(48, round(_spread(rng, 1, 48) * min(1.0, (256 * 128) / (nx * ny)))))
    c = {"kind": kind, "batch": batch, "nx": nx, "ny": ny}
    return dict(c, steps=rng.randint(1, 4)) if kind == "train" else c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _latlon(nx, ny):
    lam = torch.arange(nx, dtype=torch.float64, device="cuda") * (2.0 * math.pi / nx)
    phi = -0.5 * math.pi + (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) * (math.pi / ny)
    return lam, phi


def _waves(rng, lam, phi, kmax, n=6, even=False):
    """(f, df/dphi, (1/cos) df/dlam) of a random sum of plane waves cos(k.x + p)
    in the unit vector x, |k| <= kmax.  even: only waves whose zonal content
    has wavenumbers 0, 2, 4, ... (f(lam + pi) = f(lam)), which drive no flow
    across the poles."""
    cl, sl, cp, sp = torch.cos(lam)[None], torch.sin(lam)[None], torch.cos(phi)[:, None], torch.sin(phi)[:, None]
    f = fp = fl = 0.0
    for _ in range(n):
        k = rng.standard_normal(3)
        k *= kmax * rng.uniform(0.3, 1.0) / np.linalg.norm(k)
        a, p = float(rng.standard_normal()), float(rng.uniform(0.0, 2.0 * math.pi))
        for s in ((1.0, -1.0) if even else (1.0,)):
            kx, ky, kz = s * k[0], s * k[1], k[2]
            h = kx * cl + ky * sl
            arg = cp * h + (kz * sp + p)
            d = -a * torch.sin(arg)
            f = f + a * torch.cos(arg)
            fp = fp + d * (kz * cp - sp * h)
            fl = fl + d * (ky * cl - kx * sl)
    return f, fp, fl


def _ddlam(f):
    return (torch.roll(f, -1, 1) - torch.roll(f, 1, 1)) * (f.shape[1] / (4.0 * math.pi))


def _beyond(f, d):
    """the field one row to the north (d = 1) or south (d = -1) of each row; the
    row beyond a pole is the pole row shifted by half a circle"""
    h = f.shape[1] // 2
    return torch.cat([f[1:], torch.roll(f[-1:], h, 1)]) if d > 0 else torch.cat([torch.roll(f[:1], h, 1), f[:-1]])


def _ddphi(f):
    return (_beyond(f, 1) - _beyond(f, -1)) * (f.shape[0] / (2.0 * math.pi))


def _problem(nx, ny, seed, dt=600.0):
    """(the seven coefficient fields of Eq. 10, R) of a seeded state"""
    rng = np.random.default_rng(seed)
    lam, phi = _latlon(nx, ny)
    cp, sp = torch.cos(phi)[:, None], torch.sin(phi)[:, None]
    h = _waves(rng, lam, phi, 8.0)[0]
    depth = 8000.0 * (1.0 + 0.05 * h / h.abs().max())
    _, pp, pl = _waves(rng, lam, phi, 4.0)
    u = -pp * (40.0 / max(pp.abs().max().item(), pl.abs().max().item()))
    delta = 0.5 * dt
    alpha = (1.0 / (200.0 * dt)) * (1.0 - (0.5 * math.pi - phi.abs())[:, None] * (64.0 / (3.0 * math.pi))).clamp(min=0.0)
    c = 1.0 + delta * alpha
    b = delta * (2.0 * OMEGA * sp + u * (sp / cp) / A_EARTH)
    D = c * c + b * b
    kap, hl, hp = 0.5 * delta * GRAV * depth, _ddlam(depth), _ddphi(depth)
    q = 0.5 * delta * GRAV / D
    co = [kap * c / (D * cp), kap * b / D, -kap * b / D, kap * c * cp / D, q * (c * hl / cp + b * hp),
          q * (c * cp * hp - b * hl), (A_EARTH ** 2 / delta) * cp + torch.zeros_like(D)]
    # R: the divergence of a smooth face flux with none through the poles
    fx = _waves(rng, lam + math.pi / nx, phi, 6.0)[0]
    fy = _waves(rng, lam, phi[:-1] + 0.5 * math.pi / ny, 6.0)[0] * torch.cos(phi[:-1] + 0.5 * math.pi / ny)[:, None]
    s = A_EARTH * 8000.0 * 10.0 / max(fx.abs().max().item(), fy.abs().max().item())
    z = torch.zeros_like(fy[:1])
    R = s * ((fx - torch.roll(fx, 1, 1)) * (nx / (2.0 * math.pi)) + torch.diff(torch.cat([z, fy, z]), dim=0) * (ny / math.pi))
    return [x.contiguous() for x in co], R.contiguous()


def _members(c, seed):
    spec = [(c["nx"], c["ny"])] * c["n0"] + [(2 * c["nx"], 2 * c["ny"])] * c["n1"] + [(4 * c["nx"], 4 * c["ny"])] * c["n2"]
    return [(nx, ny, 1000 * seed + m) for m, (nx, ny) in enumerate(spec)]


def _model_state(nx, ny, seed, dt):
    """thickness, momenta, orography, relaxation rate and target of the model:
    a balanced zonal flow with smooth perturbations over 500 m of orography"""
    rng = np.random.default_rng(seed)
    lam, phi = _latlon(nx, ny)
    cp, sp = torch.cos(phi)[:, None], torch.sin(phi)[:, None]
    u0 = 20.0
    base = 8000.0 - (A_EARTH / GRAV) * (OMEGA * u0 + u0 * u0 / (2.0 * A_EARTH)) * sp * sp
    d = _waves(rng, lam, phi, 5.0, even=True)[0]
    _, pp, pl = _waves(rng, lam, phi, 3.0, even=True)
    ws = 15.0 / max(pp.abs().max().item(), pl.abs().max().item())
    m = _waves(rng, lam, phi, 4.0, even=True)[0]
    h0 = 500.0 * (m - m.min()) / (m.max() - m.min())
    depth = base + 160.0 * d / d.abs().max() - h0
    qx, qy = depth * (u0 * cp - ws * pp), depth * (ws * pl)
    alpha = (1.0 / (200.0 * dt)) * (1.0 - (0.5 * math.pi - phi.abs())[:, None] * (64.0 / (3.0 * math.pi))).clamp(min=0.0)
    return [x.contiguous() for x in (depth, qx, qy, h0, alpha + torch.zeros_like(depth), qx.clone(), qy.clone())]


def _dt(c):
    return 800.0 * 64.0 / max(c["ny"], c["nx"] // 2)


LAYERS = ((4, 32), (32, 64), (64, 64), (128, 64), (96, 32), (32, 1))


def _params(seed):
    """weights with the variance that keeps a ReLU network's signal, small biases"""
    rng = np.random.default_rng(seed)
    return np.concatenate([np.concatenate([rng.standard_normal(9 * ci * co) * math.sqrt(2.0 / (9 * ci)),
                                           0.05 * rng.standard_normal(co)]) for ci, co in LAYERS]).astype(np.float32)


def _batch(c, seed):
    """the network's inputs (a residual of unit rms, two couplings, the sine of
    the latitude) and its target, per sample"""
    nx, ny, n = c["nx"], c["ny"], c["batch"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    lam, phi = _latlon(nx, ny)
    r = torch.randn((n, ny, nx), generator=gen, device="cuda")
    w = _waves(np.random.default_rng(seed), lam, phi, 6.0)[0].float()
    x0 = torch.empty((n, 4, ny, nx), device="cuda")
    k = 0.5 + 0.4 * torch.rand((n, 1, 1), generator=gen, device="cuda")
    x0[:, 0] = 0.7 * r + 0.7 * w
    x0[:, 1] = k * (1.0 - 0.5 * torch.cos(phi).float()[None, :, None]) + 0.02 * w
    x0[:, 2] = 1.0 - x0[:, 1]
    x0[:, 3] = torch.sin(phi).float()[None, :, None]
    t = 2.0 * w + 0.5 * (r + torch.roll(r, 1, 2) + torch.roll(r, -1, 2))
    return x0, t.contiguous()


def _residual(nx, ny, seed):
    """a residual that a Krylov method meets: smooth and rough parts"""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    lam, phi = _latlon(nx, ny)
    w = _waves(np.random.default_rng(seed + 1), lam, phi, 12.0)[0]
    return 1e6 * (w + 0.3 * torch.randn((ny, nx), dtype=torch.float64, generator=gen, device="cuda"))


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("grad", "train"):
        m = sw.Model()
        sw.sw_model_set_params(m, _params(seed))
        return dict(c=c, model=m, data=[_batch(c, 100 * seed + k) for k in range(c.get("steps", 1))])
    if kind == "ensemble":
        grids, Rs, sizes = [], [], []
        for nx, ny, s in _members(c, seed):
            co, R = _problem(nx, ny, s)
            g = sw.sw_grid_create(nx, ny)
            sw.sw_elliptic_set_coeffs(g, *co)
            grids.append(g)
            Rs.append(R)
            sizes.append(R.numel())
        flat = torch.zeros(sum(sizes), dtype=torch.float64, device="cuda")
        phis = [v.view(R.shape) for v, R in zip(torch.split(flat, sizes), Rs)]
        torch.cuda.synchronize()
        return dict(c=c, grids=grids, R=Rs, flat=flat, phi=phis, stats=sw.stats_buffer(len(grids)),
                    opts=sw.sw_solve_opts_default(prec=PREC[c["prec"]], tol=1e-8))
    nx, ny = c["nx"], c["ny"]
    g = sw.sw_grid_create(nx, ny)
    if kind == "step":
        m = sw.sw_swe_create(g, _dt(c))
        return dict(c=c, grid=g, swe=m, state=_model_state(nx, ny, seed, _dt(c)),
                    out=[torch.empty((ny, nx), dtype=torch.float64, device="cuda") for _ in range(3)],
                    opts=sw.sw_solve_opts_default(prec=PREC[c["prec"]], tol=1e-8))
    co, R = _problem(nx, ny, seed)
    if kind == "solve":
        return dict(c=c, grid=g, coeffs=co, R=R, phi=torch.empty_like(R),
                    opts=sw.sw_solve_opts_default(prec=PREC[c["prec"]], tol=1e-8))
    sw.sw_elliptic_set_coeffs(g, *co)
    r = _residual(nx, ny, seed)
    if kind == "apply":
        dt = torch.float64 if c["prec"] == "fp64" else torch.float32
        x = (torch.full_like(R, 8000.0) + _residual(nx, ny, seed + 7) * 1e-4).to(dt)
        r = r.to(dt)
        torch.cuda.synchronize()
        return dict(c=c, grid=g, x=x, r=r, y=torch.empty_like(x), q=torch.empty_like(x),
                    opts=sw.sw_solve_opts_default(prec=PREC[c["prec"]]))
    m = sw.Model()
    sw.sw_model_set_params(m, _params(seed))
    return dict(c=c, grid=g, model=m, r=r.float(), e=torch.empty((ny, nx), device="cuda"))


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    s, c = state, state["c"]
    kind = c["kind"]
    if kind == "solve":
        sw.sw_elliptic_set_coeffs(s["grid"], *s["coeffs"])
        s["phi"].zero_()
        sw.sw_gcr_solve(s["grid"], s["opts"], s["R"], s["phi"])
        return s["phi"]
    if kind == "ensemble":
        s["flat"].zero_()
        sw.sw_ensemble_solve_async(s["grids"], s["opts"], s["R"], s["phi"], stats_dev=s["stats"])
        return s["flat"]
    if kind == "apply":
        sw.sw_operator_apply(s["grid"], s["x"], s["y"])
        sw.sw_precond_apply(s["grid"], s["opts"], s["r"], s["q"])
        return [s["y"], s["q"]]
    if kind == "step":
        sw.sw_swe_set_state(s["swe"], *s["state"])
        sw.sw_swe_step(s["swe"], s["opts"], c["steps"], want_stats=False)
        sw.sw_swe_get_state(s["swe"], *s["out"])
        return s["out"]
    if kind == "net":
        sw.sw_model_apply(s["model"], s["grid"], s["r"], s["e"])
        return s["e"]
    if kind == "grad":
        loss, g = sw.sw_model_loss_grad(s["model"], *s["data"][0])
        return {"loss": loss, "grad": g}
    losses = [sw.sw_model_train_step(s["model"], x0, t, lr=1e-3, weight_decay=1e-4, want_loss=(k + 1 == len(s["data"])))
              for k, (x0, t) in enumerate(s["data"])]
    return {"loss": losses[-1], "params": sw.sw_model_get_params(s["model"])}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _its(nx):
    """iterations of a solve from a zero guess to 1e-8, about"""
    return 10.0 + nx / 8.0


def work(case):
    c, kind = case, case["kind"]
    n = float(c["nx"] * c["ny"])
    if kind == "solve":       # 7 coefficient fields and R in, Phi out; about 150 operations a point an iteration
        return {"bytes": 72.0 * n, "flops": 150.0 * n * _its(c["nx"])}
    if kind == "ensemble":    # per member the face coefficients and R in, Phi out
        w = [(m[0] * m[1], _its(m[0])) for m in _members(c, 0)]
        return {"bytes": sum(72.0 * k for k, _ in w), "flops": sum(150.0 * k * i for k, i in w)}
    if kind == "apply":       # 7 face coefficients, 3 zonal factors, x and r in; y and q out
        e = 8.0 if c["prec"] == "fp64" else 4.0
        return {"bytes": 14.0 * e * n, "flops": 100.0 * n}
    if kind == "step":        # 7 fields of state in, 3 out; two solves a step, about 40 bytes of forcing a point
        return {"bytes": 80.0 * n, "flops": c["steps"] * 2 * 150.0 * n * _its(c["nx"]) / 3}
    fwd = 2.0 * 9 * n * sum(ci * co / 4.0 ** l for (ci, co), l in zip(LAYERS, (0, 1, 2, 1, 0, 0)))
    if kind == "net":         # r and three coefficient fields in, e out
        return {"bytes": 20.0 * n, "flops": fwd}
    k = c["batch"] * c.get("steps", 1)
    return {"bytes": 20.0 * n * k, "flops": 3.0 * fwd * k}


def tolerance(case):
    """Largest differences between correct implementations at the precision of
    the case, about four times those seen against exact()."""
    kind = case["kind"]
    if kind in ("solve", "ensemble"):   # the residual stops at 1e-8 of R; the operator amplifies it on larger grids
        return {"rel": 1e-6, "max": 4e-5}
    if kind == "step":
        return {"rel": 1e-9, "max": 4e-8}
    if kind == "apply":                 # FP64 sums; FP32 sums, and 16-bit storage between the stages
        return {"fp64": {"rel": 2e-13, "max": 8e-12}, "fp16": {"rel": 1e-3, "max": 4e-2}, "bf16": {"rel": 8e-3, "max": 0.3}}[case["prec"]]
    return {"rel": 2.5e-2, "max": 0.9}    # bf16 weights and activations through six layers


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _stencil(co):
    """the operator of Eq. 10 in flux form as nine weights per point, keyed by
    (rows north, points east); face values are the means of two cells, no flux
    through the pole faces.  Also P^M (Eq. 13) the same way, its diagonal's
    largest size, and the zonal coupling."""
    a11, a12, a21, a22, b1, b2, C = co
    ny, nx = C.shape
    dl, dp = 2.0 * math.pi / nx, math.pi / ny
    east = lambda f: 0.5 * (f + torch.roll(f, -1, 1))  # noqa: E731
    west = lambda f: torch.roll(f, 1, 1)  # noqa: E731

    def north(f):
        g = torch.zeros_like(f)
        g[:-1] = 0.5 * (f[:-1] + f[1:])
        return g

    def south(f):
        return torch.cat([torch.zeros_like(f[:1]), f[:-1]])

    ax, cx, bx = east(a11) / dl ** 2, east(a12) / (4 * dl * dp), east(b1) / (2 * dl)
    ay, cy, by = north(a22) / dp ** 2, north(a21) / (4 * dl * dp), north(b2) / (2 * dp)
    w = {(j, i): torch.zeros_like(C) for j in (-1, 0, 1) for i in (-1, 0, 1)}
    for cf, i0, sg in ((cx, 0, 1.0), (west(cx), -1, -1.0)):
        for i in (i0, i0 + 1):
            w[1, i] += sg * cf
            w[-1, i] -= sg * cf
    for bf, i0, sg in ((bx, 0, 1.0), (west(bx), -1, -1.0)):
        w[0, i0] += sg * bf
        w[0, i0 + 1] += sg * bf
    for yf, cf, bf, j0, sg in ((ay, cy, by, 0, 1.0), (south(ay), south(cy), south(by), -1, -1.0)):
        w[j0 + 1, 0] += sg * (yf + bf)
        w[j0, 0] += sg * (bf - yf)
        for j in (j0, j0 + 1):
            w[j, 1] += sg * cf
            w[j, -1] -= sg * cf
    pm = {k: v.clone() for k, v in w.items()}
    w[0, 1] += ax
    w[0, -1] += west(ax)
    w[0, 0] -= ax + west(ax) + C
    return w, pm, pm[0, 0].abs().max().item(), ax


def _dot(w, x):
    rows = {0: x, 1: _beyond(x, 1), -1: _beyond(x, -1)}
    return sum(v * torch.roll(rows[j], -i, 1) for (j, i), v in w.items())


def _direct(w, b):
    """solves the nine-point system by block elimination over the rows"""
    ny, nx = b.shape
    idx = torch.arange(nx, device="cuda")

    def block(j, k):
        m = torch.zeros((nx, nx), dtype=torch.float64, device="cuda")
        for i in (-1, 0, 1):
            m.index_put_((idx, (idx + i) % nx), w[k, i][j], accumulate=True)
        return m

    keep, d, g = [], None, None
    for j in range(ny):
        S, rhs = block(j, 0), b[j].clone()
        if j == 0:
            S += torch.roll(block(0, -1), nx // 2, 1)
        if j == ny - 1:
            S += torch.roll(block(j, 1), nx // 2, 1)
        if j > 0:
            low = torch.stack([w[-1, i][j] for i in (-1, 0, 1)])
            near = lambda m: sum(low[i + 1][:, None] * torch.roll(m, -i, 0) for i in (-1, 0, 1))  # noqa: E731
            S -= near(g)
            rhs -= near(d[:, None])[:, 0]
        up = block(j, 1) if j < ny - 1 else torch.zeros((nx, 0), dtype=torch.float64, device="cuda")
        sol = torch.linalg.solve(S, torch.cat([rhs[:, None], up], 1))
        d, g = sol[:, 0].clone(), sol[:, 1:]
        keep.append((d, g))
    x = torch.empty_like(b)
    for j in range(ny - 1, -1, -1):
        d, g = keep[j]
        x[j] = d if j == ny - 1 else d - g @ x[j + 1]
    return x


def _zonal(dg, of, b):
    """x of the cyclic symmetric tridiagonal system of every row: diagonal dg,
    of[i] between points i and i + 1 (the last one wraps)"""
    ny, nx = b.shape
    gam, wr = -dg[:, 0], of[:, -1]
    d = dg.clone()
    d[:, 0] -= gam
    d[:, -1] -= wr * wr / gam
    z = torch.zeros_like(b)
    z[:, 0], z[:, -1] = gam, wr
    d, o = d.t().contiguous(), of.t().contiguous()
    v = torch.stack([b.t(), z.t()], 2).contiguous()
    for i in range(1, nx):
        f = o[i - 1] / d[i - 1]
        d[i] -= f * o[i - 1]
        v[i] -= f[:, None] * v[i - 1]
    v[nx - 1] /= d[nx - 1][:, None]
    for i in range(nx - 2, -1, -1):
        v[i] = (v[i] - o[i][:, None] * v[i + 1]) / d[i][:, None]
    y, z = v[..., 0].t(), v[..., 1].t()
    t = (y[:, :1] + (wr / gam)[:, None] * y[:, -1:]) / (1.0 + z[:, :1] + (wr / gam)[:, None] * z[:, -1:])
    return y - z * t


def _precond(co, r, stages=2):
    w, pm, big, ax = _stencil(co)
    eta = 1.0 / big
    dg, of = 1.0 + eta * (ax + torch.roll(ax, 1, 1) + co[6]), -eta * ax
    q = _zonal(dg, of, -eta * r)
    for _ in range(1, stages):
        q = _zonal(dg, of, q + eta * (_dot(pm, q) - r))
    return q


def _exact_steps(c, seed):
    """the model's time steps (Eqs. 1-8) with both solves of a step done directly"""
    nx, ny, dt = c["nx"], c["ny"], _dt(c)
    P, qx, qy, h0, al, bx, by = _model_state(nx, ny, seed, dt)
    _, phi = _latlon(nx, ny)
    cp, sp = torch.cos(phi)[:, None], torch.sin(phi)[:, None]
    a, g, de, dl, dp = A_EARTH, GRAV, 0.5 * dt, 2.0 * math.pi / nx, math.pi / ny
    G, z = a * a * cp, torch.zeros((1, nx), dtype=torch.float64, device="cuda")

    def div(fl, fy):
        return (fl - torch.roll(fl, 1, 1)) / dl + torch.diff(torch.cat([z, fy, z]), dim=0) / dp

    def carried(f, U, V):
        Uf, Vf = 0.5 * (U + torch.roll(U, -1, 1)), 0.5 * (V[:-1] + V[1:])
        return div(Uf.clamp(min=0) * f + Uf.clamp(max=0) * torch.roll(f, -1, 1), Vf.clamp(min=0) * f[:-1] + Vf.clamp(max=0) * f[1:])

    up = vp = None
    for _ in range(c["steps"]):
        u, v = qx / P, qy / P
        up, vp = (u, v) if up is None else (up, vp)
        U, V = a * (1.5 * u - 0.5 * up), a * cp * (1.5 * v - 0.5 * vp)
        fn = 2.0 * OMEGA * sp + u * (sp / cp) / a
        px = qx + de * (-(g / (a * cp)) * P * _ddlam(P + h0) + fn * qy - al * (qx - bx))
        py = qy + de * (-(g / a) * P * _ddphi(P + h0) - fn * qx - al * (qy - by))
        hx, hy = px - (dt / G) * carried(px, U, V), py - (dt / G) * carried(py, U, V)
        cc, b = 1.0 + de * al, de * (2.0 * OMEGA * sp + (2.0 * u - up) * (sp / cp) / a)
        D = cc * cc + b * b
        ps = P
        for _ in range(2):
            kap, sl, sn = 0.5 * de * g * ps, _ddlam(ps + h0), _ddphi(ps + h0)
            q = 0.5 * de * g / D
            co = [kap * cc / (D * cp), kap * b / D, -kap * b / D, kap * cc * cp / D, q * (cc * sl / cp + b * sn),
                  q * (cc * cp * sn - b * sl), G / de + torch.zeros_like(P)]
            X0 = hx + de * al * bx - de * (0.5 * g / (a * cp)) * ps * _ddlam(h0)
            Y0 = hy + de * al * by - de * (0.5 * g / a) * ps * _ddphi(h0)
            Fx, Fy = a * (qx + (cc * X0 + b * Y0) / D), a * cp * (qy + (cc * Y0 - b * X0) / D)
            w = _stencil(co)[0]
            rhs = div(0.5 * (Fx + torch.roll(Fx, -1, 1)), 0.5 * (Fy[:-1] + Fy[1:])) - co[6] * P - _dot(w, P)
            inc = _direct(w, rhs)
            last, ps = ps, P + inc
        P = ps
        X = X0 - de * (0.5 * g / (a * cp)) * (P * sl + last * _ddlam(P))
        Y = Y0 - de * (0.5 * g / a) * (P * sn + last * _ddphi(P))
        qx, qy, up, vp = (cc * X + b * Y) / D, (cc * Y - b * X) / D, u, v
    return [P, qx, qy]


def _conv(x, w, b):
    W = x.shape[-1]
    x = torch.cat([torch.roll(x[:, :, :1], W // 2, 3), x, torch.roll(x[:, :, -1:], W // 2, 3)], 2)
    x = torch.cat([x[..., -1:], x, x[..., :1]], 3)
    return torch.nn.functional.conv2d(x, w, b)


def _unflat(p):
    out, at = [], 0
    for ci, co in LAYERS:
        out.append((p[at:at + 9 * ci * co].view(co, ci, 3, 3), p[at + 9 * ci * co:at + 9 * ci * co + co]))
        at += 9 * ci * co + co
    return out


def _network(p, x):
    L, relu = _unflat(p), torch.relu
    pool = lambda t: torch.nn.functional.avg_pool2d(t, 2)  # noqa: E731
    up = lambda t: t.repeat_interleave(2, 2).repeat_interleave(2, 3)  # noqa: E731
    a1 = relu(_conv(x, *L[0]))
    a2 = relu(_conv(pool(a1), *L[1]))
    a3 = relu(_conv(pool(a2), *L[2]))
    a4 = relu(_conv(torch.cat([up(a3), a2], 1), *L[3]))
    a5 = relu(_conv(torch.cat([up(a4), a1], 1), *L[4]))
    return _conv(a5, *L[5])[:, 0]


def _loss_grad(p, x0, t):
    """the mean squared error over the batch and its gradient, four samples at a time"""
    p = p.detach().requires_grad_(True)
    loss, grad = 0.0, torch.zeros_like(p)
    for k in range(0, x0.shape[0], 4):
        part = (_network(p, x0[k:k + 4].double()) - t[k:k + 4].double()).square().sum() / t.numel()
        grad += torch.autograd.grad(part, p)[0]
        loss += float(part)
    return loss, grad


def exact(case, seed):
    c, kind = case, case["kind"]
    with torch.backends.cudnn.flags(enabled=False):
        if kind == "solve":
            if c["nx"] > 1024:
                return None          # the direct solution takes minutes
            co, R = _problem(c["nx"], c["ny"], seed)
            return _direct(_stencil(co)[0], R)
        if kind == "ensemble":
            out = []
            for nx, ny, s in _members(c, seed):
                if nx > 256:         # the largest members: too many direct solutions
                    return None
                co, R = _problem(nx, ny, s)
                out.append(_direct(_stencil(co)[0], R).reshape(-1))
            return torch.cat(out)
        if kind == "apply":
            co, R = _problem(c["nx"], c["ny"], seed)
            dt = torch.float64 if c["prec"] == "fp64" else torch.float32
            x = (torch.full_like(R, 8000.0) + _residual(c["nx"], c["ny"], seed + 7) * 1e-4).to(dt).double()
            r = _residual(c["nx"], c["ny"], seed).to(dt).double()
            return [_dot(_stencil(co)[0], x), _precond(co, r)]
        if kind == "step":
            return _exact_steps(c, seed) if c["nx"] <= 512 else None
        p = torch.from_numpy(_params(seed)).cuda().double()
        if kind == "net":
            nx, ny = c["nx"], c["ny"]
            co, _ = _problem(nx, ny, seed)
            w, _, _, ax = _stencil(co)
            r = _residual(nx, ny, seed).float().double()
            d = w[0, 0].abs()
            ay = torch.zeros_like(d)
            ay[:-1] = 0.5 * (co[3][:-1] + co[3][1:]) * (ny / math.pi) ** 2
            ays = torch.cat([torch.zeros_like(ay[:1]), ay[:-1]])
            s = r.square().mean().sqrt()
            sin = torch.sin(_latlon(nx, ny)[1])[:, None] + torch.zeros_like(r)
            x0 = torch.stack([r / s, (ax + torch.roll(ax, 1, 1)) / d, (ay + ays) / d, sin])
            return s * _network(p, x0[None])[0] / d
        if c["batch"] * c["nx"] * c["ny"] * c.get("steps", 1) > 64 * 256 * 128:
            return None              # minutes of FP64 convolutions
        if kind == "grad":
            loss, g = _loss_grad(p, *_batch(c, 100 * seed))
            return {"loss": loss, "grad": g}
        m, v = torch.zeros_like(p), torch.zeros_like(p)
        bias = torch.cat([torch.cat([torch.zeros(9 * ci * co), torch.ones(co)]) for ci, co in LAYERS]).cuda().bool()
        for k in range(c["steps"]):
            loss, g = _loss_grad(p, *_batch(c, 100 * seed + k))
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            mh, vh = m / (1.0 - 0.9 ** (k + 1)), v / (1.0 - 0.999 ** (k + 1))
            p = p.detach() - 1e-3 * (mh / (vh.sqrt() + 1e-8) + torch.where(bias, 0.0, 1e-4) * p.detach())
        return {"loss": loss, "params": p}
