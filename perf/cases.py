"""Workloads of the travel-time and ray-Born paths, each one call sequence of a
user's program through the package's public functions.

A case is a dict of plain values; ``kind`` names the call sequence:

  forward    travel times of one emitter's rays at given angles (rt_tof_forward)
  link       ray linking of all pairs, cold (rt_link)
  link_grad  ray linking, then the retraced gradient (rt_link + rt_tof_adjoint)
  autograd   the differentiable travel times and their backward pass (tof)
  rows       linking that records the system-matrix rows, gradient from them
             (rt_link_rows + rt_tof_adjoint_rows), cold or from given angles
  linearise  explicit system matrix and SART sweeps on it (rt_path_matrix +
             inversion.sart_solve)
  batch      many uneven problems, linked with gradient in one call (rt_batch_run)
  maps       per-transducer travel-time and amplitude maps (rtborn_maps)
  born       ray-Born data of a perturbation and the adjoint of a residual
             (rtborn_apply + rtborn_adjoint)

Geometry follows the repository's configurations: a centred nx x ny grid of
spacing h, a ring of n_tx transducers at 0.45 of the shorter side, step h / 10,
fans traced at h / 2. Media are a 1500 m/s background with smooth Gaussian
inclusions ("gauss"), 40 smoothed ellipses of 1400-1600 m/s ("breast"), or one
sound speed of about that ("uniform").
"""
import math

import torch

import paper_2511_18511_gb300 as rt
from paper_2511_18511_gb300 import inversion
from paper_2511_18511_gb300.phantoms import Grid

DEV = "cuda"
STEP_FLOPS = {"rk4": 219, "heun": 125}      # per ray step, bilinear sampler
BSPLINE_STEP_FLOPS = 387
FAN_STEP_FLOPS = 403                        # per step of a map fan (with its paraxial ray)


def _tof(name, kind, nx, ny, h, n_tx, medium, **kw):
    case = {"name": name, "kind": kind, "nx": nx, "ny": ny, "h": h, "n_tx": n_tx, "medium": medium,
            "precision": "fp32c", "integrator": "rk4", "interpolator": "bilinear", "fan_rays": 256, "warm": False}
    case.update(kw)
    return case


def listed():
    return [
        # one shot of a small ring at known angles: the smallest call, launches and latency
        _tof("forward_128_ring64_shot", "forward", 128, 128, 0.5, 64, "gauss"),
        # the small all-pairs link of a quick look or a test rig
        _tof("link_128_ring64", "link", 128, 128, 0.5, 64, "gauss"),
        # the first gradient of an inversion at full size: cold link with recorded rows + adjoint
        _tof("rows_breast_1024_ring512", "rows", 1024, 1024, 0.2, 512, "breast", fan_rays=768),
        # a later gradient of an inversion on an odd-sized grid and ring, started from the
        # straight-ray angles of the homogeneous model before it
        _tof("rows_warm_531x517_ring203", "rows", 531, 517, 0.2, 203, "gauss", warm=True),
        # the differentiable travel times inside somebody's own torch optimisation
        _tof("autograd_512_ring256", "autograd", 512, 512, 0.2, 256, "gauss"),
        # the paper's second field sampler
        _tof("bspline_384_ring128", "link_grad", 384, 384, 0.2, 128, "gauss", interpolator="bspline"),
        # double precision, the reference accuracy of the library
        _tof("fp64_128_ring64", "link_grad", 128, 128, 0.5, 64, "gauss", precision="fp64"),
        # an inversion's first linearisation: the explicit matrix of the homogeneous starting
        # model and SART sweeps on it, the paper's Heun integrator
        _tof("linearise_192_ring96", "linearise", 192, 192, 0.4, 96, "uniform", integrator="heun", sweeps=10),
        # a throughput job: several patients' uneven slices in one call
        {"name": "batch_8", "kind": "batch", "instances": 8, "pick": 4, "side_max": 768, "ring_max": 256},
        # ray-Born background maps of a full-size grid, one eighth of the 512 fans
        {"name": "maps_1024_tx64", "kind": "maps", "nx": 1024, "ny": 1024, "h": 0.2, "n_tx": 64, "lossy": False},
        # one ray-Born product and its adjoint at full grid size
        {"name": "born_1024_ring384_f4", "kind": "born", "nx": 1024, "ny": 1024, "h": 0.2, "n_tx": 384, "freqs": 4,
         "lossy": False},
        # the same pair at the small configuration, with power-law absorption
        {"name": "born_128_ring64_f8_lossy", "kind": "born", "nx": 128, "ny": 128, "h": 0.5, "n_tx": 64, "freqs": 8,
         "lossy": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "link", "link_grad", "autograd", "rows", "linearise", "batch", "maps", "born"])
    if kind == "batch":
        return {"kind": kind, "instances": rng.randint(2, 8), "pick": rng.randint(0, 10 ** 6),
                "side_max": rng.choice([384, 512, 768]), "ring_max": rng.choice([128, 192, 256])}
    n = _log_int(rng, 96, 1024)
    nx, ny = n, max(96, n - rng.randint(0, n // 16))
    h = rng.choice([0.2, 0.25, 0.4, 0.5])
    if kind == "maps":
        return {"kind": kind, "nx": nx, "ny": ny, "h": h, "n_tx": _log_int(rng, 8, 64), "lossy": rng.random() < 0.3}
    if kind == "born":
        n_tx, freqs = _log_int(rng, 24, 384), rng.randint(1, 8)
        while n_tx * n_tx * freqs > 384 * 384 * 4:
            freqs -= 1
        return {"kind": kind, "nx": nx, "ny": ny, "h": h, "n_tx": n_tx, "freqs": freqs, "lossy": rng.random() < 0.3}
    case = {"kind": kind, "nx": nx, "ny": ny, "h": h, "n_tx": _log_int(rng, 24, 320),
            "medium": rng.choice(["gauss", "breast"]), "precision": "fp32c",
            "integrator": rng.choice(["rk4", "rk4", "heun"]), "interpolator": "bilinear",
            "fan_rays": rng.choice([0, 128, 256, 256, 384]), "warm": rng.random() < 0.3}
    if kind == "link_grad":
        case["precision"], case["interpolator"] = rng.choice([("fp64", "bilinear"), ("fp32c", "bspline"),
                                                              ("fp32c", "bspline"), ("fp32c", "bilinear")])
        if case["precision"] == "fp64":        # a double-precision march costs about thirty single ones
            case["nx"] = case["ny"] = rng.randint(96, 160)
            case["n_tx"] = rng.randint(24, 72)
    elif kind == "linearise":                  # the matrix holds every cell visit of every ray
        case["nx"] = case["ny"] = _log_int(rng, 96, 384)
        case["n_tx"] = _log_int(rng, 24, 128)
        case["medium"], case["sweeps"] = "uniform", rng.randint(4, 16)
    if case["nx"] > 384 and case["fan_rays"] == 0:     # straight starts are for the small problems
        case["fan_rays"] = 256
    if kind in ("rows", "autograd"):           # these calls march by their fixed integrator or sampler
        case["integrator"] = "rk4"
    return case


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device="cpu")
    g.manual_seed(int(seed))
    return g


def _uniform(g, n, lo, hi):
    return (lo + (hi - lo) * torch.rand(n, generator=g, dtype=torch.float64)).to(DEV)


def _radius(nx, ny, h):
    return 0.45 * min(nx, ny) * h


def _axes(nx, ny, h):
    x = (torch.arange(nx, dtype=torch.float64, device=DEV) - (nx - 1) / 2.0) * h
    y = (torch.arange(ny, dtype=torch.float64, device=DEV) - (ny - 1) / 2.0) * h
    return x, y


def _blur(img, sigma):
    """Gaussian blur of sigma nodes, rows of the kernel normalised at the edges."""
    def k(n):
        i = torch.arange(n, dtype=torch.float64, device=DEV)
        w = torch.exp(-((i[:, None] - i[None, :]) ** 2) / (2.0 * sigma * sigma))
        return w / w.sum(1, keepdim=True)
    return k(img.shape[0]) @ img @ k(img.shape[1]).T


def _medium(kind, nx, ny, h, g):
    """Sound speed [ny, nx] in m/s."""
    R = _radius(nx, ny, h)
    x, y = _axes(nx, ny, h)
    X, Y = x[None, :], y[:, None]
    if kind == "uniform":
        return (torch.ones(ny, nx, dtype=torch.float64, device=DEV) * _uniform(g, 1, 1480.0, 1520.0)).contiguous()
    if kind == "gauss":
        m, sc = 3, R / 30.0
        rad, ang = 0.6 * R * torch.sqrt(_uniform(g, m, 0, 1)), _uniform(g, m, 0, 2 * math.pi)
        sig = _uniform(g, m, 3.0 * sc, 6.0 * sc)
        amp = torch.where(_uniform(g, m, 0, 1) < 0.5, -0.03, 0.03)
        rel = torch.zeros(ny, nx, dtype=torch.float64, device=DEV)
        for k in range(m):
            d2 = (X - rad[k] * torch.cos(ang[k])) ** 2 + (Y - rad[k] * torch.sin(ang[k])) ** 2
            rel += amp[k] * torch.exp(-d2 / (2.0 * sig[k] ** 2))
        return (1500.0 * (1.0 + rel)).contiguous()
    m, sc = 40, R / 95.0
    cv = _uniform(g, m, 1400.0, 1600.0)
    ax, ay = _uniform(g, m, 2.0 * sc, 15.0 * sc), _uniform(g, m, 2.0 * sc, 15.0 * sc)
    rot = _uniform(g, m, 0.0, math.pi)
    rad, ang = 70.0 * sc * torch.sqrt(_uniform(g, m, 0, 1)), _uniform(g, m, 0, 2 * math.pi)
    img = torch.full((ny, nx), 1480.0, dtype=torch.float64, device=DEV)
    for k in range(m):
        dx, dy = X - rad[k] * torch.cos(ang[k]), Y - rad[k] * torch.sin(ang[k])
        u = dx * torch.cos(rot[k]) + dy * torch.sin(rot[k])
        v = -dx * torch.sin(rot[k]) + dy * torch.cos(rot[k])
        img = torch.where((u / ax[k]) ** 2 + (v / ay[k]) ** 2 <= 1.0, cv[k], img)
    return _blur(img, math.hypot(1.0, 3.0) * sc / h).contiguous()


def _ring(n_tx, R):
    a = 2.0 * math.pi * torch.arange(n_tx, dtype=torch.float64, device=DEV) / n_tx
    return torch.stack([R * torch.cos(a), R * torch.sin(a)], dim=1).contiguous()


def _all_pairs(n_tx):
    e = torch.arange(n_tx, device=DEV).repeat_interleave(n_tx - 1)
    r = torch.arange(n_tx - 1, device=DEV).repeat(n_tx)
    return e, r + (r >= e).long()


def _measured(tx, e, r, g):
    """Travel times (us) as measured: the straight path at 1500 m/s, off by up to 0.5 %."""
    d = (tx[e] - tx[r]).norm(dim=1)
    return (d / 1.5 * (1.0 + 0.005 * torch.sin(_uniform(g, d.numel(), 0.0, 2 * math.pi)))).contiguous()


def _straight(tx, e, r):
    d = tx[r] - tx[e]
    return torch.atan2(d[:, 1], d[:, 0]).contiguous()


def _problem(nx, ny, h, n_tx, medium, g):
    R = _radius(nx, ny, h)
    tx = _ring(n_tx, R)
    return rt.Problem(Grid(nx, ny, h), _medium(medium, nx, ny, h, g), tx, R)


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "batch":
        return {"case": case, "instances": _batch(case, seed)}
    nx, ny, h, n_tx = case["nx"], case["ny"], case["h"], case["n_tx"]
    st = {"case": case}
    if kind == "maps":
        st["prob"] = p = _problem(nx, ny, h, n_tx, "breast", g)
        # fans dense enough that neighbouring rays stay within a grid step at the far side
        st["fan"] = 64 * math.ceil(4.0 * math.pi * p.ring_radius / h / 64)
        if case["lossy"]:
            st["alpha0"] = 2.0e-8 * (1.0 + 20.0 * (p.c / 1500.0 - 1.0).abs())
        return st
    if kind == "born":
        return {**st, **_born(case, g)}
    st["prob"] = p = _problem(nx, ny, h, n_tx, case["medium"], g)
    st["ds"], st["fan_ds"] = h / 10.0, h / 2.0
    e, r = _all_pairs(n_tx)
    if kind == "forward":                      # the receivers of one emitter
        shot = int(torch.randint(n_tx, (1,), generator=g))
        e, r = e[e == shot], r[e == shot]
        p.pairs = torch.stack([e, r], dim=1).to(torch.int32).contiguous()
    st["theta"] = _straight(p.tx, e, r)
    st["t_meas"] = _measured(p.tx, e, r, g)
    if kind == "rows":
        st["rows"] = rt.Rows.create(p)
    return st


def _batch_sizes(case):
    g = _gen(case["pick"])
    for _ in range(case["instances"]):
        n = int(torch.randint(1, case["side_max"] // 128 + 1, (1,), generator=g)) * 128
        n_tx = int(torch.randint(32, case["ring_max"] + 1, (1,), generator=g))
        yield n, n_tx


def _batch(case, seed):
    out = []
    for k, (n, n_tx) in enumerate(_batch_sizes(case)):
        g = _gen(seed * 64 + k)
        p = _problem(n, n, 0.2, n_tx, "gauss", g)
        e, r = _all_pairs(n_tx)
        out.append(rt.BatchInstance.create(p, _measured(p.tx, e, r, g)))
    return out


def _born(case, g):
    nx, ny, h, n_tx = case["nx"], case["ny"], case["h"], case["n_tx"]
    R = _radius(nx, ny, h)
    tx = _ring(n_tx, R)
    x, y = _axes(nx, ny, h)
    inside = (x[None, :] ** 2 + y[:, None] ** 2) < R * R
    T = torch.empty(n_tx, ny, nx, dtype=torch.float32, device=DEV)
    A = torch.empty_like(T)
    L = torch.empty_like(T) if case["lossy"] else None
    ph = _uniform(g, 4, 0.0, 2 * math.pi)
    # first-arrival times of mild refraction, geometric amplitudes, unreached outside the ring
    slow = 1.0 / 1.5 * (1.0 + 0.01 * torch.sin(3.0 * x / R + ph[0])[None, :] * torch.sin(2.0 * y / R + ph[1])[:, None])
    for t in range(n_tx):
        r = torch.sqrt((x[None, :] - tx[t, 0]) ** 2 + (y[:, None] - tx[t, 1]) ** 2)
        bend = 1.0 + 0.004 * torch.sin(0.05 * r + ph[2] + 2.0 * math.pi * t / n_tx)
        T[t] = torch.where(inside, r * slow * bend, math.inf).float()
        A[t] = torch.where(inside, torch.rsqrt(r.clamp(min=h)), 0.0).float()
        if L is not None:
            L[t] = torch.where(inside, 2.0e-11 * r * (1.0 + 0.2 * torch.sin(0.03 * r + ph[3])), 0.0).float()
    maps = rt.BornMaps(Grid(nx, ny, h), R, T, A, L, 1.3 if case["lossy"] else 1.0)
    dc = torch.where(inside, 5.0 * torch.randn(ny, nx, generator=g, dtype=torch.float64).to(DEV), 0.0).float()
    f = [0.5 + 1.0 * k / max(1, case["freqs"] - 1) for k in range(case["freqs"])]
    d = torch.view_as_complex(torch.randn(len(f), n_tx, n_tx, 2, generator=g).to(DEV))
    return {"maps": maps, "dc": dc.contiguous(), "f": f, "d": d.contiguous()}


# ---------------------------------------------------------------- one pass

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        b = rt.rt_batch_run(st["instances"], 0.02, fan_ds=0.1)
        return [{"theta": i.theta, "tof": i.tof, "hit": i.hit, "status": i.status, "iters": i.iters, "g": i.g_c}
                for i in b]
    if kind == "maps":
        p = st["prob"]
        m = rt.rtborn_maps(p, p.grid.h / 10.0, st["fan"], alpha0=st.get("alpha0"), y=1.3)
        return {"T": m.T, "A": m.A} if m.L is None else {"T": m.T, "A": m.A, "L": m.L}
    if kind == "born":
        return {"d": rt.rtborn_apply(st["maps"], st["f"], st["dc"]),
                "dc": rt.rtborn_adjoint(st["maps"], st["f"], st["d"])}
    p, ds = st["prob"], st["ds"]
    how = {"precision": case["precision"], "integrator": case["integrator"], "interpolator": case["interpolator"]}
    start = {"theta0": st["theta"] if case["warm"] else None, "fan_rays": case["fan_rays"]}
    if kind == "forward":
        t, hit = rt.rt_tof_forward(p, st["theta"], ds, **how)
        return {"tof": t, "hit": hit}
    if kind == "link":
        return rt.rt_link(p, ds, fan_ds=st["fan_ds"], **start, **how)
    if kind == "link_grad":
        out = rt.rt_link(p, ds, fan_ds=st["fan_ds"], **start, **how)
        return {**out, "g": rt.rt_tof_adjoint(p, out["theta"], out["tof"], ds, tof_ref=st["t_meas"], **how)}
    if kind == "autograd":
        c = p.c.detach().requires_grad_(True)
        t = rt.tof(c, p, ds, precision=case["precision"], **start)
        loss = 0.5 * ((t - st["t_meas"]) ** 2).sum()
        (g,) = torch.autograd.grad(loss, c)
        return {"tof": t.detach(), "loss": loss.detach(), "g": g}
    if kind == "rows":
        out = rt.rt_link_rows(p, ds, st["rows"], fan_ds=st["fan_ds"], **start)
        g = rt.rt_tof_adjoint_rows(p, st["rows"], out["theta"], out["tof"], ds, tof_ref=st["t_meas"])
        return {**out, "len": st["rows"].len, "g": g}
    row_ptr, col, val = rt.rt_path_matrix(p, st["theta"], ds, **how)
    op = inversion.csr_operator(row_ptr, col, val, p.c.numel())
    s = inversion.sart_solve(op, st["t_meas"], (1000.0 / p.c).reshape(-1), case["sweeps"])
    return {"row_ptr": row_ptr, "col": col, "val": val, "s": s}


# ---------------------------------------------------------------- what a pass cannot do without

def _ray_steps(pairs, R, ds):
    return pairs * 4.0 * R / math.pi / ds          # the mean chord of a ring is 4 R / pi


def _tof_work(nx, ny, h, pairs, fan, integrator, interpolator, grad, grad_marches):
    R, ds = _radius(nx, ny, h), h / 10.0
    per = BSPLINE_STEP_FLOPS if interpolator == "bspline" else STEP_FLOPS[integrator]
    steps = _ray_steps(pairs, R, ds) * (2 if grad_marches else 1) + _ray_steps(fan, R, h / 2.0)
    b = 8.0 * nx * ny * (2 if grad else 1) + pairs * (8 + 8 + 16 + 8 + (8 if grad else 0))
    return {"bytes": b, "flops": steps * per}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for n, n_tx in _batch_sizes(case):
            w = _tof_work(n, n, 0.2, n_tx * (n_tx - 1), n_tx * 256, "rk4", "bilinear", True, False)
            total = {k: total[k] + w[k] for k in total}
        return total
    nx, ny, h, n_tx = case["nx"], case["ny"], case["h"], case["n_tx"]
    R = _radius(nx, ny, h)
    if kind == "maps":
        rays = n_tx * 64 * math.ceil(4.0 * math.pi * R / h / 64)
        maps = 3 if case["lossy"] else 2
        return {"bytes": 8.0 * nx * ny * (2 if case["lossy"] else 1) + 4.0 * maps * n_tx * nx * ny,
                "flops": rays * 2.0 * R * (2.0 / math.pi) / (h / 10.0) * FAN_STEP_FLOPS}
    if kind == "born":
        n_in, maps = math.pi * (R / h) ** 2, 3 if case["lossy"] else 2
        # both products: each map read once, the symmetric half of n_tx^2 complex sums per node
        return {"bytes": 2.0 * (4.0 * maps * n_tx * n_in + 4.0 * nx * ny + 8.0 * case["freqs"] * n_tx * n_tx),
                "flops": 2.0 * 4.0 * n_tx * n_tx * n_in * case["freqs"]}
    pairs = n_tx * (n_tx - 1)
    fan = n_tx * case["fan_rays"] if not case["warm"] else 0
    if kind == "forward":
        return _tof_work(nx, ny, h, n_tx - 1, 0, case["integrator"], case["interpolator"], False, False)
    if kind == "linearise":
        w = _tof_work(nx, ny, h, pairs, 0, case["integrator"], case["interpolator"], False, False)
        nnz = pairs * 4.0 * 4.0 * R / math.pi / h * 4.0 / math.pi    # four nodes per cell visit
        passes = 2 * case["sweeps"] + 2
        return {"bytes": w["bytes"] + 12.0 * nnz * (1 + passes), "flops": w["flops"] + 2.0 * nnz * passes}
    return _tof_work(nx, ny, h, pairs, fan, case["integrator"], case["interpolator"], kind != "link", False)


# ---------------------------------------------------------------- the same results in 64 bits

class _Field:
    """Bilinear sampling of c, its gradient and the slowness, in double precision."""

    def __init__(self, p):
        c = 1e-3 * p.c
        self.h, self.x0, self.y0, self.nx, self.ny = p.grid.h, p.grid.x0, p.grid.y0, p.grid.nx, p.grid.ny
        gy, gx = torch.gradient(c, spacing=self.h)
        self.F = torch.stack([c, gx, gy, 1.0 / c]).reshape(4, -1)

    def at(self, x, y):
        u, v = (x - self.x0) / self.h, (y - self.y0) / self.h
        i = u.floor().clamp(0, self.nx - 2)
        j = v.floor().clamp(0, self.ny - 2)
        tx, ty = u - i, v - j
        k = (j * self.nx + i).long()
        nodes = torch.stack([k, k + 1, k + self.nx, k + self.nx + 1])
        w = torch.stack([(1 - tx) * (1 - ty), tx * (1 - ty), (1 - tx) * ty, tx * ty])
        return (self.F[:, nodes] * w).sum(1), nodes, w

    def rhs(self, x, y, dx, dy):
        (c, gx, gy, _), _, _ = self.at(x, y)
        gd = gx * dx + gy * dy
        return dx, dy, (gd * dx - gx) / c, (gd * dy - gy) / c

    def step(self, z, H, heun):
        def go(k, a):
            return [p + a * q for p, q in zip(z, k)]
        k1 = self.rhs(*z)
        if heun:
            k2 = self.rhs(*go(k1, H))
            n = [p + 0.5 * H * (a + b) for p, a, b in zip(z, k1, k2)]
        else:
            k2 = self.rhs(*go(k1, 0.5 * H))
            k3 = self.rhs(*go(k2, 0.5 * H))
            k4 = self.rhs(*go(k3, H))
            n = [p + H / 6.0 * (a + 2.0 * (b + c) + d) for p, a, b, c, d in zip(z, k1, k2, k3, k4)]
        r = torch.sqrt(n[2] ** 2 + n[3] ** 2)
        return [n[0], n[1], n[2] / r, n[3] / r]


def _trace(F, R, ds, xe, theta, xr, heun, sink=None):
    """Fixed-step march to the ring: (travel time, hit); sink(nodes, weights, rays) takes
    the trapezoid weights of every sample point."""
    z = [xe[:, 0].clone(), xe[:, 1].clone(), torch.cos(theta), torch.sin(theta)]
    ids = torch.arange(theta.numel(), device=DEV)
    last = [torch.zeros_like(theta) for _ in range(4)]
    T = torch.zeros_like(theta)
    s_prev = None
    m = 0
    while ids.numel():
        f, nodes, w = F.at(z[0], z[1])
        s = f[3]
        if m:
            T.index_add_(0, ids, 0.5 * ds * (s_prev + s))
        if sink is not None:
            sink(nodes, w * (0.5 * ds if m == 0 else ds), ids)
        n = F.step(z, ds, heun)
        out = n[0] ** 2 + n[1] ** 2 >= R * R
        if bool(out.any()):
            for a, b in zip(last, z):
                a[ids[out]] = b[out]
            keep = ~out
            ids, n, s = ids[keep], [a[keep] for a in n], s[keep]
        z, s_prev = n, s
        m += 1
        if m > 8.0 * R / ds:
            return None
    # the last step, shortened to end on the ring
    t = torch.full_like(theta, 0.5 * ds)
    for _ in range(8):
        e = F.step(last, t, heun)
        r = torch.sqrt(e[0] ** 2 + e[1] ** 2)
        t = (t - (r - R) / ((e[0] * e[2] + e[1] * e[3]) / r)).clamp(0.0, ds)
    e = F.step(last, t, heun)
    fl, nl, wl = F.at(last[0], last[1])
    fe, ne, we = F.at(e[0], e[1])
    corr = e[2] * (xr[:, 0] - e[0]) + e[3] * (xr[:, 1] - e[1])
    T += 0.5 * t * (fl[3] + fe[3]) + fe[3] * corr
    if sink is not None:
        every = torch.arange(theta.numel(), device=DEV)
        sink(nl, wl * (0.5 * (t - ds)), every)
        sink(ne, we * (0.5 * t + corr), every)
    return T, torch.stack([e[0], e[1]], dim=1)


def _linked(F, R, ds, xe, xr, theta, heun):
    """Launch angles whose rays end at xr, by the secant rule from the given angles."""
    def miss(th):
        _, hit = _trace(F, R, ds, xe, th, xr, heun)
        return torch.atan2(xr[:, 0] * hit[:, 1] - xr[:, 1] * hit[:, 0], (xr * hit).sum(1))
    m0 = miss(theta)
    th = theta - 0.5 * m0
    for _ in range(5):
        m = miss(th)
        den = m - m0
        new = torch.where((den != 0) & (m.abs() > 1e-13), th - m * (th - theta) / den, th)
        theta, m0, th = th, m, new
    lo = torch.atan2(xe[:, 1], xe[:, 0]) + 0.5 * math.pi     # angles lie in the inward half-turn from here
    return lo + torch.remainder(th - lo, 2.0 * math.pi)


def exact(case, seed):
    kind = case["kind"]
    if kind == "born":
        n_in = math.pi * (_radius(case["nx"], case["ny"], case["h"]) / case["h"]) ** 2
        return _born_exact(prepare(case, seed)) if case["n_tx"] ** 2 * n_in * case["freqs"] < 6e11 else None
    # a march in torch costs about a hundred kernels a step; the others' steps are too many
    if kind not in ("forward", "link", "link_grad") or case["interpolator"] != "bilinear":
        return None
    R = _radius(case["nx"], case["ny"], case["h"])
    traces = 1 if kind == "forward" else 8
    if traces * 2.0 * R / (case["h"] / 10.0) * max(1.0, case["n_tx"] ** 2 / 3e4) > 1.5e4 or case["medium"] != "gauss":
        return None
    st = prepare(case, seed)
    p, heun = st["prob"], case["integrator"] == "heun"
    F = _Field(p)
    e, r = _all_pairs(p.n_tx) if p.pairs is None else (p.pairs[:, 0].long(), p.pairs[:, 1].long())
    xe, xr, theta = p.tx[e], p.tx[r], st["theta"]
    if kind == "forward":
        T, hit = _trace(F, R, st["ds"], xe, theta, xr, heun)
        return {"tof": T, "hit": hit}
    theta = _linked(F, R, st["ds"], xe, xr, theta, heun)
    T, _ = _trace(F, R, st["ds"], xe, theta, xr, heun)
    out = {"theta": theta, "tof": T, "hit": xr, "status": None, "iters": None}
    if kind == "link":
        return out
    g = torch.zeros(p.c.numel(), dtype=torch.float64, device=DEV)
    w = T - st["t_meas"]
    _trace(F, R, st["ds"], xe, theta, xr, heun,
           lambda nodes, a, ids: g.index_add_(0, nodes.reshape(-1), (a * w[ids]).reshape(-1)))
    return {**out, "g": -1000.0 * g.reshape(p.c.shape) / p.c ** 2}


def _born_exact(st):
    maps, dc, d = st["maps"], st["dc"].double().reshape(-1), st["d"].to(torch.complex128)
    n_tx, h = maps.n_tx, maps.grid.h
    keep = torch.isfinite(maps.T[0]).reshape(-1).nonzero().reshape(-1)
    off = ~torch.eye(n_tx, dtype=torch.bool, device=DEV)
    data = torch.zeros(len(st["f"]), n_tx, n_tx, dtype=torch.complex128, device=DEV)
    back = torch.zeros(dc.numel(), dtype=torch.float64, device=DEV)
    for part in keep.split(65536):
        T = maps.T.reshape(n_tx, -1)[:, part].double()
        A = maps.A.reshape(n_tx, -1)[:, part].double()
        L = None if maps.L is None else maps.L.reshape(n_tx, -1)[:, part].double()
        for k, f in enumerate(st["f"]):
            om = 2.0 * math.pi * f
            amp = A if L is None else A * torch.exp(-((om * 1e6) ** maps.y) * L)
            E = torch.polar(amp, om * T)
            w = om * om * h * h
            data[k] += w * (E * dc[part]) @ E.T
            back[part] += w * (E.conj() * ((d[k] * off) @ E.conj())).sum(0).real
    return {"d": data * off, "dc": back.reshape(st["dc"].shape)}
