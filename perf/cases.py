"""The work that a user of the DD-4DVar library has it do, as timed cases.

Every case is one pass through a public entry point of ``paper_2205_06649_gb300``
on a twin experiment: a shallow-water truth on the sphere (Gaussian height
bumps in geostrophic balance), a background with errors of sigma_b, and
observations of the truth run with errors of sigma_o.  The sizes are those of
the workloads in this repository (small, ragged, medium, differentiation,
batching, one time window of the large one).

``exact`` restates the method in plain torch in 64 bits: the box model with
frozen lateral ghosts, the local functionals by reverse-mode differentiation,
Gauss-Newton products by forward- and reverse-mode, the global model and the
Turkel-Zwas functional.
"""
from __future__ import annotations

import math

import numpy as np
import torch

RADIUS, GRAVITY, OMEGA = 6.371e6, 9.81, 7.292e-5
LAT = 80.0            # walls at +-80 degrees
H_REF = 4000.0
SIGMA_B = (5.0, 0.1, 0.1)
SIGMA_O = (1.0, 0.05, 0.05)
RF_PASSES = 4
F64 = torch.float64


def _case(name, kind, nlon, nlat, nsteps, P1=1, P2=1, Q=1, o=4, ot=4, uneven=False, obs="random", n_obs=0.05,
          every=8, corr=3.0, precision=0, ckpt=0, host=False, iters=20, p=1, q=1, alpha=0.0):
    """obs "grid": n_obs is the share of the grid points observed at every observed level (all of h, u, v;
    h alone for the small workload); "random": n_obs observations at fractional positions over the window."""
    c = dict(kind=kind, nlon=nlon, nlat=nlat, nsteps=nsteps, P1=P1, P2=P2, Q=Q, o=o, ot=ot, uneven=uneven, obs=obs,
             n_obs=n_obs, every=every, corr=corr, precision=precision, ckpt=ckpt, host=host, iters=iters, p=p, q=q,
             alpha=alpha)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: J and grad J of 8 small boxes, diagonal B (the small workload); latency and launches
        _case("eval small f64", "eval", 32, 16, 16, 2, 2, 2, 2, 2, obs="grid", n_obs=0.1, every=4, corr=0.0),
        # odd and uneven boxes, called with host arrays as a C or numpy program does (the ragged workload)
        _case("eval ragged f32 host", "eval", 70, 38, 30, 3, 2, 3, 3, 3, uneven=True, n_obs=1500, every=3, corr=2.0,
              precision=1, host=True),
        # the ordinary evaluation in each precision: 64 equal boxes (the medium workload)
        _case("eval medium f64", "eval", 256, 128, 128, 4, 4, 4, obs="grid"),
        _case("eval medium f32", "eval", 256, 128, 128, 4, 4, 4, obs="grid", precision=1),
        # differentiable J in a torch program, trajectory checkpointed every 16 steps (the differentiation workload)
        _case("autograd differentiation f32", "grad", 512, 256, 256, 8, 4, 4, obs="grid", precision=1, ckpt=16),
        # many uneven boxes in one batched evaluation, each precision (the batching workload, diagonal B)
        _case("eval batching f64", "eval", 1024, 512, 512, 8, 8, 8, 4, 8, uneven=True, n_obs=100000, corr=0.0),
        _case("eval batching f32", "eval", 1024, 512, 512, 8, 8, 8, 4, 8, uneven=True, n_obs=100000, corr=0.0,
              precision=1),
        # one 128-step window of the large workload's 256 boxes, 1/8 of its observations, correlated B
        _case("eval large window f32", "eval", 2048, 1024, 128, 16, 16, 1, 8, 8, uneven=True, n_obs=125000, every=4,
              precision=1),
        # a whole outer iteration of Algorithm 1: 20 batched L-BFGS iterations and the exchange (medium workload)
        _case("outer step medium f64", "outer", 256, 128, 128, 4, 4, 4, obs="grid"),
        # one Gauss-Newton product (tangent-linear and adjoint sweep), the inner step of the other local solver
        _case("gauss-newton product medium f64", "gn", 256, 128, 128, 4, 4, 4, obs="grid"),
        # the undecomposed functional and gradient in the paper's Turkel-Zwas discretisation
        _case("turkel-zwas eval medium", "tz", 256, 128, 128, obs="grid", corr=0.0, p=2, q=1, alpha=0.5),
        # the global model run that makes truth and background trajectories
        _case("global run 512x256", "forward", 512, 256, 256),
    ]


def draw(rng):
    """One more case of the same ranges: box cores of 12..150 x 7..75 points in 1..8 blocks per axis, 1..8 windows
    of 11..72 steps, up to 1.5e8 points x steps; global runs of 24..512 longitudes."""
    kind = rng.choice(["eval", "eval", "eval", "eval", "grad", "outer", "gn", "tz", "forward"])
    span = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    precision = rng.randrange(2)
    if kind in ("tz", "forward"):
        nlon = span(24, 512)
        nlat = max(12, int(nlon * rng.uniform(0.4, 0.6)))
        nsteps = min(span(8, 256), max(8, int(1.5e7 // (nlon * nlat))))
        return _case(None, kind, nlon, nlat, nsteps, n_obs=max(8, nlon * nlat // 20), every=rng.choice([2, 4, 8]),
                     corr=0.0, p=rng.randint(1, 3), q=rng.randint(1, 2), alpha=rng.choice([0.0, 1.0 / 3.0, 0.5]))
    most = 1.5e8 if kind in ("eval", "grad") else 6e6
    while True:
        P1, P2, Q = rng.choice([1, 2, 3, 4, 6, 8]), rng.choice([1, 2, 3, 4, 6, 8]), rng.choice([1, 2, 3, 4, 8])
        core_x, core_y, core_t = span(12, 150), span(7, 75), span(11, 72)
        o, ot = rng.choice([2, 3, 4]), rng.choice([2, 3, 4])
        uneven = rng.random() < 0.5
        if core_x < 5 * o:
            core_x += 5 * o
        if core_y < 3 * o:
            core_y += 3 * o
        nlon, nlat, nsteps = P1 * core_x + rng.randrange(P1), P2 * core_y + rng.randrange(P2), Q * core_t
        if P1 == 1:
            nlon = min(nlon, 160)
        steps = P1 * P2 * Q * (core_x + 2 * o) * (core_y + 2 * o) * (core_t + 2 * ot)
        if steps <= most and (P1 > 1 or nlon >= 8) and core_t > 3.4 * ot and nlon * nlat * nsteps < 3e8:
            break
    every = rng.choice([2, 4, 8])
    n = int(min(200000, max(20, 0.05 * nlon * nlat * (nsteps / every + 1))))
    ckpt = 16 if kind == "grad" and rng.random() < 0.5 else 0
    return _case(None, kind, nlon, nlat, nsteps, P1, P2, Q, o, ot, uneven=uneven, n_obs=n, every=every,
                 corr=rng.choice([0.0, 2.0, 3.0]), precision=precision, ckpt=ckpt,
                 host=kind == "eval" and steps < 1e6 and rng.random() < 0.5, iters=rng.choice([5, 10, 20]))


# ---- inputs, from the seed alone -------------------------------------------------------------------------------------

def _rows(nlat, dev):
    th0, dth = math.radians(-LAT), math.radians(2 * LAT) / nlat
    return th0 + (torch.arange(nlat, dtype=F64, device=dev) + 0.5) * dth, dth


class _Grid:
    def __init__(self, nlon, nlat, dev):
        self.nlon, self.nlat = nlon, nlat
        self.th, self.dth = _rows(nlat, dev)
        self.dlam = 2.0 * math.pi / nlon
        self.cos = torch.cos(self.th)
        self.A = 1.0 / (2.0 * RADIUS * self.cos * self.dlam)
        self.f = 2.0 * OMEGA * torch.sin(self.th)
        self.tau = torch.tan(self.th) / RADIUS
        self.Bth = 1.0 / (2.0 * RADIUS * self.dth)


_MIRROR = torch.tensor([1.0, 1.0, -1.0], dtype=F64)


def _tend(z, A, f, tau, cos, cos_e, Bth):
    """Tendencies at the interior of z [..., 3, ny+2, nx+2]; row constants [..., ny, 1], cos_e [..., ny+2, 1]."""
    h, u, v = z[..., 0, :, :], z[..., 1, :, :], z[..., 2, :, :]
    mid, c = slice(1, -1), (Ellipsis, slice(1, -1), slice(1, -1))
    uc, vc = u[c], v[c]
    dx = lambda a: a[..., mid, 2:] - a[..., mid, :-2]  # noqa: E731
    dy = lambda a: a[..., 2:, mid] - a[..., :-2, mid]  # noqa: E731
    fu = f + tau * uc
    Fu = -A * uc * dx(u) - Bth * vc * dy(u) + fu * vc - GRAVITY * A * dx(h)
    Fv = -A * uc * dx(v) - Bth * vc * dy(v) - fu * uc - GRAVITY * Bth * dy(h)
    Fh = -A * dx(h * u) - (Bth / cos) * dy(h * v * cos_e)
    return torch.stack([Fh, Fu, Fv], dim=-3)


def _rk3(x, F, dt, ext):
    """ext(state, stage): the state with its ghost ring at that stage's time."""
    x1 = x + dt * F(ext(x, 0))
    x2 = 0.75 * x + 0.25 * (x1 + dt * F(ext(x1, 1)))
    return x / 3.0 + (2.0 / 3.0) * (x2 + dt * F(ext(x2, 2)))


def _global_levels(g, x, dt, nsteps):
    """The global model's levels 0..nsteps, one after the other."""
    mir = _MIRROR.to(x.device)[:, None, None]
    ce = torch.cat([g.cos[:1], g.cos, g.cos[-1:]])[:, None]
    F = lambda z: _tend(z, g.A[:, None], g.f[:, None], g.tau[:, None], g.cos[:, None], ce, g.Bth)  # noqa: E731

    def ext(s, _):
        s = torch.cat([s[..., -1:], s, s[..., :1]], dim=-1)
        return torch.cat([s[:, :1] * mir, s, s[:, -1:] * mir], dim=1)

    yield x
    for _ in range(nsteps):
        x = _rk3(x, F, dt, ext)
        yield x


def _truth(c, g, gen, dev):
    """Bumps of 50 m and 8 degrees on 4000 m at rest, winds in geostrophic balance (f floored near the equator)."""
    r = torch.rand(9, generator=gen, dtype=F64, device=dev).cpu().numpy()
    lam = torch.arange(g.nlon, dtype=F64, device=dev)[None, :] * g.dlam
    th = g.th[:, None]
    sig = math.radians(8.0)
    h = torch.full((g.nlat, g.nlon), H_REF, dtype=F64, device=dev)
    hy, hx = torch.zeros_like(h), torch.zeros_like(h)
    for k in range(3):
        lc, tc = 2 * math.pi * r[3 * k], math.radians(20.0 + 40.0 * r[3 * k + 1]) * (1 if r[3 * k + 2] > 0.5 else -1)
        K = (torch.sin(th) * math.sin(tc) + torch.cos(th) * math.cos(tc) * torch.cos(lam - lc)).clamp(-1 + 1e-12, 1 - 1e-12)
        d = torch.arccos(K)
        e = 50.0 * torch.exp(-d * d / (2 * sig * sig))
        s = e * d / torch.sin(d) / (sig * sig)
        h = h + e
        hy = hy + s * (torch.cos(th) * math.sin(tc) - torch.sin(th) * math.cos(tc) * torch.cos(lam - lc))
        hx = hx - s * torch.cos(th) * math.cos(tc) * torch.sin(lam - lc)
    f = (2 * OMEGA * torch.sin(th)).abs().clamp(min=2 * OMEGA * math.sin(math.radians(10.0)))
    f = torch.where(th < 0, -f, f)
    return torch.stack([h, -GRAVITY / (f * RADIUS) * hy, GRAVITY / (f * RADIUS * torch.cos(th)) * hx])


def _smooth(x, ell):
    """Noise of unit variance correlated over ell cells, periodic in longitude."""
    s = ell / math.sqrt(2.0)
    r = min(int(math.ceil(4 * s)), min(x.shape[-2:]) - 1)
    k = torch.exp(-torch.arange(-r, r + 1, dtype=F64, device=x.device) ** 2 / (2 * s * s))
    k = k / k.square().sum().sqrt()
    y = torch.nn.functional.pad(x[:, None], (r, r, 0, 0), mode="circular")
    y = torch.nn.functional.conv2d(y, k[None, None, None, :])
    y = torch.nn.functional.pad(y, (0, 0, r, r), mode="reflect")
    return torch.nn.functional.conv2d(y, k[None, None, :, None])[:, 0]


def _cuts(n, parts, uneven, r, least):
    if not uneven or parts == 1:
        return np.array([k * n // parts for k in range(parts + 1)], dtype=np.int32)
    share = 0.7 + 0.6 * r
    size = np.maximum(least, np.floor(share / share.sum() * n).astype(int))
    while size.sum() != n:
        k = int(np.argmin(size)) if size.sum() < n else int(np.argmax(size))
        size[k] += 1 if size.sum() < n else -1
    return np.concatenate([[0], np.cumsum(size)]).astype(np.int32)


def _inputs(c, seed):
    dev = "cuda"
    gen = torch.Generator(dev).manual_seed(seed)
    g = _Grid(c["nlon"], c["nlat"], dev)
    xt = _truth(c, g, gen, dev)
    width = min(RADIUS * float(g.cos.min()) * g.dlam, RADIUS * g.dth)
    dt = float("%.3g" % (0.45 * width / (math.sqrt(GRAVITY * float(xt[0].max())) + float(xt[1:].abs().max()))))
    xi = torch.randn(xt.shape, generator=gen, dtype=F64, device=dev)
    if c["corr"]:
        xi = _smooth(xi, c["corr"])
    I = dict(g=g, xt=xt, dt=dt, xb=xt + torch.tensor(SIGMA_B, dtype=F64, device=dev)[:, None, None] * xi)
    if c["kind"] == "forward":
        return I
    r = torch.rand(3 * 16, generator=gen, dtype=F64, device=dev).cpu().numpy()
    for k, (key, n, parts, least) in enumerate((("lon", c["nlon"], c["P1"], max(2, 2 * c["o"])),
                                                ("lat", c["nlat"], c["P2"], max(2, 2 * c["o"])),
                                                ("t", c["nsteps"], c["Q"], 2 * c["ot"] + 1))):
        I[key] = _cuts(n, parts, c["uneven"], r[16 * k:16 * k + parts], least)
    # observation sites
    levels = torch.arange(0, c["nsteps"] + 1, c["every"], device=dev)
    if c["obs"] == "grid":
        var = (0,) if c["corr"] == 0.0 and c["nlon"] <= 32 else (0, 1, 2)
        n = max(1, int(round(c["n_obs"] * c["nlon"] * c["nlat"])))
        at = [torch.randperm(c["nlon"] * c["nlat"], generator=gen, device=dev)[:n].sort().values for _ in levels]
        lv = torch.cat([torch.full((n * len(var),), int(t), device=dev) for t in levels])
        vr = torch.cat([torch.full((n,), v, device=dev) for v in var] * len(levels))
        pos = torch.cat([a for a in at for _ in var])
        fi, fj = (pos % c["nlon"]).to(F64), (pos // c["nlon"]).to(F64)
    else:
        n = int(c["n_obs"])
        u = torch.rand(4, n, generator=gen, dtype=F64, device=dev)
        lv = levels[(u[0] * len(levels)).long()].sort().values
        vr = (u[1] * 3).long()
        fi, fj = u[2] * c["nlon"], u[3] * (c["nlat"] - 1)
    so = torch.tensor(SIGMA_O, dtype=F64, device=dev)[vr]
    y = torch.empty(len(lv), dtype=F64, device=dev)
    count = torch.bincount(lv, minlength=c["nsteps"] + 1).cpu().numpy()
    lo = 0
    for t, x in enumerate(_global_levels(g, xt, dt, c["nsteps"])):
        if count[t]:
            s = slice(lo, lo + int(count[t]))
            y[s] = _bilinear(x, vr[s], fi[s], fj[s])
            lo += int(count[t])
    y = y + so * torch.randn(len(y), generator=gen, dtype=F64, device=dev)
    I.update(lv=lv, vr=vr, fi=fi, fj=fj, y=y, so=so)
    # controls at which a minimiser evaluates, and a direction
    n = sum(b["n"] for b in _boxes(c, I)) if c["kind"] != "tz" else 3 * c["nlon"] * c["nlat"]
    I["w"] = 0.3 * torch.randn(n, generator=gen, dtype=F64, device=dev)
    if c["kind"] == "gn":
        I["p"] = torch.randn(n, generator=gen, dtype=F64, device=dev)
    return I


def _bilinear(x, var, fi, fj):
    i0, j0 = fi.floor().long(), fj.floor().long()
    di, dj = fi - i0, fj - j0
    i1, j1 = (i0 + 1) % x.shape[-1], (j0 + 1).clamp(max=x.shape[-2] - 1)
    return ((1 - dj) * (1 - di) * x[var, j0, i0] + (1 - dj) * di * x[var, j0, i1]
            + dj * (1 - di) * x[var, j1, i0] + dj * di * x[var, j1, i1])


def prepare(case, seed):
    import paper_2205_06649_gb300 as dd
    c = dict(case)
    I = _inputs(c, seed)
    S = dict(case=c)
    ctx = dd.Context(c["nlon"], c["nlat"], I["dt"], c["nsteps"], precision=c["precision"])
    S["ctx"] = ctx
    if c["kind"] == "forward":
        S["x0"] = I["xt"].contiguous()
        return S
    ctx.set_background(I["xb"].cpu().numpy())
    ctx.set_background_error(SIGMA_B, c["corr"], RF_PASSES)
    ctx.set_observations(*[I[k].cpu().numpy() for k in ("lv", "vr", "fi", "fj", "y", "so")])
    if c["kind"] == "tz":
        S["w"] = I["w"].cpu().numpy()
        return S
    ctx.set_decomposition(c["P1"], c["P2"], c["Q"], c["o"], c["o"], c["ot"], I["lon"], I["lat"], I["t"],
                          ckpt_k=c["ckpt"])
    S["w"] = I["w"].cpu().numpy() if c["host"] else I["w"]
    if c["kind"] == "gn":
        S["p"] = I["p"]
    if c["kind"] == "outer":
        S["solver"] = dd.solver_defaults(max_local_iters=c["iters"])
        S["w0"] = torch.zeros_like(I["w"])
    return S


def run(S):
    c, ctx = S["case"], S["ctx"]
    if c["kind"] == "forward":
        return {"traj": ctx.forward(S["x0"])}
    if c["kind"] == "tz":
        J, g = ctx.tz_eval(c["p"], c["q"], c["alpha"], S["w"])
        return {"J": J, "grad": g}
    if c["kind"] == "gn":
        return {"Ap": ctx.gn_hessvec(S["w"], S["p"])}
    if c["kind"] == "grad":
        from paper_2205_06649_gb300.autograd import dd4dvar_J
        w = S["w"].detach().requires_grad_(True)
        J = dd4dvar_J(w, ctx)
        J.sum().backward()
        return {"J": J.detach(), "grad": w.grad}
    if c["kind"] == "outer":   # the first outer iteration: from the background state and zero controls
        ctx.reset_exchange()
        ctx.set_controls(S["w0"])
        stats = ctx.outer_step(S["solver"])
        return {"w": ctx.get_controls(), "analysis": ctx.analysis(), "J_sum": stats.J_sum, "dw_inf": stats.dw_inf}
    J, g = ctx.eval(S["w"])
    return {"J": J, "grad": g}


# ---- what a pass cannot do without -----------------------------------------------------------------------------------

def _axes(c, I=None):
    """(start, length) of the extended blocks per axis; without inputs, those of equal cuts."""
    out = []
    for key, n, parts, o, wrap in (("lon", c["nlon"], c["P1"], c["o"], True), ("lat", c["nlat"], c["P2"], c["o"], False),
                                   ("t", c["nsteps"], c["Q"], c["ot"], False)):
        cut = I[key] if I is not None else [k * n // parts for k in range(parts + 1)]
        ax = []
        for k in range(parts):
            a, b = int(cut[k]), int(cut[k + 1])
            if parts > 1:
                a, b = a - o, b + o
                if not wrap:
                    a, b = max(0, a), min(n, b)
            ax.append((a % n if wrap else a, b - a))
        out.append(ax)
    return out


def work(case):
    """Flops: 141 a point and step for the model (3 tendencies of 35, stage combinations 36) and 228 for its adjoint;
    bytes: inputs and outputs once (controls, background at the window starts, frozen ghosts, targets at shared points,
    observations, J and gradient)."""
    c = case
    el = 4 if c["precision"] else 8
    N = c["nlon"] * c["nlat"]
    if c["kind"] == "forward":
        return {"bytes": 24.0 * N * (c["nsteps"] + 2), "flops": 141.0 * N * c["nsteps"]}
    n_lv = c["nsteps"] // c["every"] + 1
    n_obs = c["n_obs"] * N * 3 * n_lv if c["obs"] == "grid" else c["n_obs"]
    if c["kind"] == "tz":
        return {"bytes": 24.0 * N * 3 + 40.0 * n_obs, "flops": 2 * 450.0 * N * c["nsteps"]}
    X, Y, T = _axes(c)
    steps = pts = ghosts = shared = 0
    for _, nx in X:
        for _, ny in Y:
            core = max(1, nx - 4 * c["o"] * (c["P1"] > 1)) * max(1, ny - 4 * c["o"] * (c["P2"] > 1))
            for _, L in T:
                steps += nx * ny * L
                pts += 3 * nx * ny
                ghosts += 6 * (nx + ny) * (L + 1)
                shared += 3 * (nx * ny - core) * (L + 1)
    byt = pts * (8 + 8 + 8) + (ghosts + shared) * el + 56.0 * n_obs
    flops = 369.0 * steps
    if c["kind"] == "gn":
        byt, flops = byt + 8 * pts, flops + (228.0 + 141.0) * steps
    if c["kind"] == "outer":
        byt, flops = byt * c["iters"] + 24.0 * N * (c["nsteps"] + 1), flops * c["iters"]
    return {"bytes": float(byt), "flops": float(flops)}


# ---- the method in plain torch, 64 bits ------------------------------------------------------------------------------

def _boxes(c, I):
    X, Y, T = _axes(c, I)
    return [dict(i0=X[p1][0], nx=X[p1][1], j0=Y[p2][0], ny=Y[p2][1], a=T[q][0], L=T[q][1], n=3 * X[p1][1] * Y[p2][1],
                 p1=p1, p2=p2, q=q)
            for q in range(c["Q"]) for p2 in range(c["P2"]) for p1 in range(c["P1"])]


def _filter(n, ell, dev):
    """The recursive filter c (F^T F)^N on a line of n points, as a matrix."""
    E = 2.0 * RF_PASSES / (ell * ell)
    a = 1.0 + E - math.sqrt(E * (E + 2.0))

    def apply(x, times):
        for _ in range(times):
            for order in (range(len(x)), range(len(x) - 1, -1, -1)):
                q = np.zeros(x.shape[1])
                for i in order:
                    q = a * q + (1.0 - a) * x[i]
                    x[i] = q
        return x

    half = int(40 * ell) + 60
    e = np.zeros((2 * half + 1, 1))
    e[half] = 1.0
    amp = 1.0 / math.sqrt(apply(e, 2 * RF_PASSES)[half, 0])
    return torch.tensor(amp * apply(np.eye(n), RF_PASSES), dtype=F64, device=dev)


def _residuals(c, I, B, group, w):
    """J_s terms of boxes of one shape as weighted residuals: J = 1/2 w.w + 1/2 r.r (per box) with w [b, 3, ny, nx]."""
    g, dev, dt = I["g"], w.device, I["dt"]
    b0 = group[0]
    nx, ny, L, nb = b0["nx"], b0["ny"], b0["L"], len(group)
    per = c["P1"] == 1
    cols = torch.tensor([[(b["i0"] + k) % g.nlon for k in range(-1, nx + 1)] for b in group], device=dev)
    rows = torch.tensor([[min(max(b["j0"] + k, 0), g.nlat - 1) for k in range(-1, ny + 1)] for b in group], device=dev)
    lev = torch.tensor([b["a"] for b in group], device=dev)
    con = [v[rows[:, 1:-1]][:, :, None] for v in (g.A, g.f, g.tau, g.cos)]
    F = lambda z: _tend(z, *con, g.cos[rows][:, :, None], g.Bth)  # noqa: E731
    full = lambda l: B[(lev + l)[:, None, None, None], torch.arange(3, device=dev)[None, :, None, None],  # noqa: E731
                       rows[:, None, :, None], cols[:, None, None, :]]
    mir = _MIRROR.to(dev)[None, :, None, None]

    def ring(l):
        z = full(l)
        return z[:, :, :1, 1:-1], z[:, :, -1:, 1:-1], z[:, :, 1:-1, :1], z[:, :, 1:-1, -1:]

    def extend(s, gh):
        S, N, W, E = gh
        if per:
            W, E = s[..., -1:], s[..., :1]
        if b0["j0"] == 0:
            S = s[:, :, :1] * mir
        if b0["j0"] + ny == g.nlat:
            N = s[:, :, -1:] * mir
        zero = torch.zeros(nb, 3, 1, 1, dtype=F64, device=dev)
        return torch.cat([torch.cat([zero, S, zero], 3), torch.cat([W, s, E], 3), torch.cat([zero, N, zero], 3)], 2)

    v = w
    if c["corr"]:
        v = torch.einsum("rs,bvsk,lk->bvrl", _filter(ny, c["corr"], dev), v, _filter(nx, c["corr"], dev))
    sb = torch.tensor(SIGMA_B, dtype=F64, device=dev)[None, :, None, None]
    x = full(0)[:, :, 1:-1, 1:-1] + sb * v
    traj, gh = [x], ring(0)
    for l in range(L):
        nxt = ring(l + 1)
        mean = tuple(0.5 * (p + q) for p, q in zip(gh, nxt))
        x = _rk3(x, F, dt, lambda s, k: extend(s, (gh, nxt, mean)[k]))
        traj.append(x)
        gh = nxt
    x = torch.stack(traj, 1)                                    # [b, L+1, 3, ny, nx]
    # overlap: every other box that covers the point pulls towards the background
    band = lambda n, lo, hi: (torch.arange(n, device=dev) < lo).double() + (torch.arange(n, device=dev) >= n - hi).double()  # noqa: E731
    o2 = 2 * c["o"]
    cx = 1 + band(nx, o2 * (not per), o2 * (not per))
    cy = 1 + band(ny, o2 * (b0["p2"] > 0), o2 * (b0["p2"] < c["P2"] - 1))
    ct = torch.stack([1 + band(L + 1, (2 * c["ot"] + 1) * (b["q"] > 0), (2 * c["ot"] + 1) * (b["q"] < c["Q"] - 1)) for b in group])
    cnt = ct[:, :, None, None] * cy[None, None, :, None] * cx - 1
    bg = torch.stack([full(l)[:, :, 1:-1, 1:-1] for l in range(L + 1)], 1)
    r = [(cnt.sqrt()[:, :, None] * (x - bg) / sb[:, None]).reshape(nb, -1)]
    # observations
    i0, j0 = I["fi"].floor().long(), I["fj"].floor().long()
    di, dj = I["fi"] - i0, I["fj"] - j0
    out = []
    for k, b in enumerate(group):
        s = _sees(b, I, g, i0, j0, di, dj).nonzero()[:, 0]
        k0, r0 = (i0[s] - b["i0"]) % g.nlon, j0[s] - b["j0"]
        k1 = torch.where(di[s] != 0, (i0[s] + 1 - b["i0"]) % g.nlon, k0)
        r1 = torch.where(dj[s] != 0, r0 + 1, r0)
        l, vr, a, d = I["lv"][s] - b["a"], I["vr"][s], di[s], dj[s]
        X = x[k]
        hx = ((1 - d) * (1 - a) * X[l, vr, r0, k0] + (1 - d) * a * X[l, vr, r0, k1]
              + d * (1 - a) * X[l, vr, r1, k0] + d * a * X[l, vr, r1, k1])
        out.append((hx - I["y"][s]) / I["so"][s] / I["seen"][s].sqrt())
    return r[0], out


def _sees(b, I, g, i0, j0, di, dj):
    k0, k1 = (i0 - b["i0"]) % g.nlon, (i0 + 1 - b["i0"]) % g.nlon
    lon = (k0 < b["nx"]) & ((di == 0) | (k1 < b["nx"]))
    lat = (j0 >= b["j0"]) & (j0 < b["j0"] + b["ny"]) & ((dj == 0) | (j0 + 1 < b["j0"] + b["ny"]))
    return lon & lat & (I["lv"] >= b["a"]) & (I["lv"] <= b["a"] + b["L"])


def _groups(c, I):
    B = torch.stack(list(_global_levels(I["g"], I["xb"], I["dt"], c["nsteps"])))
    boxes, off = _boxes(c, I), 0
    i0, j0 = I["fi"].floor().long(), I["fj"].floor().long()
    seen = torch.zeros(len(i0), dtype=F64, device=i0.device)
    sets = {}
    for k, b in enumerate(boxes):
        b.update(off=off, s=k)
        off += b["n"]
        seen += _sees(b, I, I["g"], i0, j0, I["fi"] - i0, I["fj"] - j0)
        sets.setdefault((b["nx"], b["ny"], b["L"], b["p2"] > 0, b["p2"] < c["P2"] - 1), []).append(b)
    I["seen"] = seen
    return B, list(sets.values())


def _pack(group, flat):
    return torch.stack([flat[b["off"]:b["off"] + b["n"]].reshape(3, b["ny"], b["nx"]) for b in group])


def _exact_boxes(c, I):
    B, groups = _groups(c, I)
    n_sub = c["P1"] * c["P2"] * c["Q"]
    J, out = torch.zeros(n_sub, dtype=F64), torch.zeros(I["w"].numel(), dtype=F64)
    for group in groups:
        w = _pack(group, I["w"])
        if c["kind"] == "gn":
            import torch.autograd.forward_ad as fw
            with torch.no_grad(), fw.dual_level():
                r, obs = _residuals(c, I, B, group, fw.make_dual(w, _pack(group, I["p"])))
                tr = fw.unpack_dual(r).tangent
                to = [fw.unpack_dual(o).tangent for o in obs]
        w.requires_grad_(True)
        r, obs = _residuals(c, I, B, group, w)
        if c["kind"] == "gn":
            dot = (r * tr).sum() + sum((o * t).sum() for o, t in zip(obs, to) if t is not None)
            res = _pack(group, I["p"]) + torch.autograd.grad(dot, w)[0]
        else:
            Js = 0.5 * w.square().sum((1, 2, 3)) + 0.5 * r.square().sum(1) + 0.5 * torch.stack([o.square().sum() for o in obs])
            res = torch.autograd.grad(Js.sum(), w)[0]
            for b, v in zip(group, Js.detach().cpu()):
                J[b["s"]] = v
        for b, v in zip(group, res.cpu()):
            out[b["off"]:b["off"] + b["n"]] = v.reshape(-1)
        del r, obs, res
    return {"Ap": out} if c["kind"] == "gn" else {"J": J, "grad": out}


def _exact_tz(c, I):
    g, dev, p, q, al = I["g"], I["w"].device, c["p"], c["q"], c["alpha"]
    sl, st = 1.0 / (2 * RADIUS * g.dlam), g.Bth
    m = _MIRROR.to(dev)[:, None, None]
    ev = lambda r: torch.cat([r[:q].flip(0), r, r[-q:].flip(0)])[:, None]  # noqa: E731
    ce, fe, te = ev(g.cos), ev(g.f), ev(g.tau)
    cos, f, tau = g.cos[:, None], g.f[:, None], g.tau[:, None]

    def at(a, di, dj):
        a = a[q + dj:q + dj + g.nlat]
        return torch.roll(a, -di, -1) if di else a

    def F(x):
        z = torch.cat([x[:, :q].flip(1) * m, x, x[:, -q:].flip(1) * m], 1)
        h, u, v = z
        hc, uc, vc, vk = at(h, 0, 0), at(u, 0, 0), at(v, 0, 0), v * ce
        Ce = (fe + u * te)
        cu = (1 - al) * at(Ce, 0, 0) * vc + 0.5 * al * (at(Ce * v, p, 0) + at(Ce * v, -p, 0))
        cv = (1 - al) * at(Ce, 0, 0) * uc + 0.5 * al * (at(Ce * u, 0, q) + at(Ce * u, 0, -q))
        dx, dy = lambda a, s=1: at(a, s, 0) - at(a, -s, 0), lambda a, s=1: at(a, 0, s) - at(a, 0, -s)
        Fu = -sl * uc / cos * dx(u) - st * vc * dy(u) - sl * GRAVITY / (p * cos) * dx(h, p) + cu
        Fv = -sl * uc / cos * dx(v) - st * vc * dy(v) - st * GRAVITY / q * dy(h, q) - cv
        du = (1 - al) * dx(u, p) + 0.5 * al * (at(u, p, q) - at(u, -p, q) + at(u, p, -q) - at(u, -p, -q))
        dv = (1 - al) * dy(vk, q) + 0.5 * al * (at(vk, p, q) - at(vk, p, -q) + at(vk, -p, q) - at(vk, -p, -q))
        Fh = -(sl * uc / cos * dx(h) + st * vc * dy(h) + sl * hc / (p * cos) * du + st * hc / (q * cos) * dv)
        return torch.stack([Fh, Fu, Fv])

    w = I["w"].clone().requires_grad_(True)
    x = I["xb"] + torch.tensor(SIGMA_B, dtype=F64, device=dev)[:, None, None] * w.reshape(3, g.nlat, g.nlon)
    J = 0.5 * w.square().sum()
    for t in range(c["nsteps"] + 1):
        if t:
            x = _rk3(x, F, I["dt"], lambda s, _: s)
        s = (I["lv"] == t).nonzero()[:, 0]
        if len(s):
            J = J + 0.5 * ((_bilinear(x, I["vr"][s], I["fi"][s], I["fj"][s]) - I["y"][s]) / I["so"][s]).square().sum()
    return {"J": float(J.detach()), "grad": torch.autograd.grad(J, w)[0].cpu().numpy()}


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "outer":
        return None      # an evaluation takes seconds here, an outer iteration has over 20
    if c["kind"] in ("eval", "grad", "gn"):
        X, Y, T = _axes(c)
        shapes = min(len(X), 8 if c["uneven"] else 2) * min(len(Y), 8 if c["uneven"] else 3) * min(len(T), 8 if c["uneven"] else 2)
        if shapes * max(L for _, L in T) > 3000 or c["nlon"] * c["nlat"] * c["nsteps"] > 4e7:
            return None  # many distinct boxes: over 20 s of separate passes
    I = _inputs(c, seed)
    if c["kind"] == "forward":
        return {"traj": torch.stack(list(_global_levels(I["g"], I["xt"], I["dt"], c["nsteps"])))}
    if c["kind"] == "tz":
        return _exact_tz(c, I)
    with torch.enable_grad():
        return _exact_boxes(c, I)
