"""The workloads this library's speed is judged by, each one pass through the public binding.

Snapshots are synthetic stand-ins for a flow solver's fields (a cylinder in a potential flow
with a vortex-blob wake, an undulating swimmer, a Lamb-Oseen vortex), generated on the GPU
from a seed.  ``listed()`` holds the cases, ``draw()`` more of the same ranges, ``prepare()``
what a program holds before the call (fields, points, a plan with its captured step), ``run()``
one pass, ``work()`` the bytes and operations of a pass and ``exact()`` the same results in
64 bits by the direct sum (evaluated as a zero-padded convolution on uniform grids).
"""
import functools
import math

import numpy as np
import torch

from paper_1610_04398_gb300 import api, synth

LAMBDA, NU = 1e4, 1e-4
RHO_H = math.exp(math.pi / 4 - 1.5 - 0.5 * math.log(2.0))  # clamp of |x - x'| in units of h


def listed():
    return [
        # the smallest snapshot of a swimmer batch, one captured step: launches and latency count
        _grid("swimmer_256_step", "graph", "swimmer", 256, 12, 0.7, 128, 0.5, 4096),
        # a mid-size snapshot by separate calls with the plan's default tile and surface
        # acceptance, the source kept: a program that is being developed
        _grid("swimmer_512_calls", "calls", "swimmer", 512, 16, 0.5, 16, 0.0, 2048),
        # the headline benchmark: a 2048^2 cylinder snapshot at the autotuned setting
        _grid("cylinder_2048_step", "graph", "cylinder", 2048, 12, 0.75, 128, 0.5, 2048),
        # the same grid at a strict setting (order 20, theta 0.5, near field on the FP32 cores)
        _grid("cylinder_2048_strict_step", "graph", "cylinder", 2048, 20, 0.5, 16, 0.0, 2048),
        # the largest grid served, at the server's order and acceptance
        _grid("cylinder_4096_step", "graph", "cylinder", 4096, 12, 0.6, 128, 0.0, 4096),
        # uneven swimmer snapshots in one launch
        {"name": "swimmer_batch_16", "mode": "batch", "flow": "swimmer", "count": 16, "nmin": 256, "nmax": 2048,
         "order": 12, "theta": 0.7, "tile": 128, "theta_surface": 0.5, "npts": 4096, "precision": "mixed"},
        # the FP64 path: the small vortex of the accuracy checks, and a cylinder at full accuracy
        _grid("lamb_oseen_128_fp64", "calls", "vortex", 128, 20, 0.5, 16, 0.0, 256, "fp64"),
        _grid("cylinder_1024_fp64", "calls", "cylinder", 1024, 20, 0.5, 16, 0.0, 2048, "fp64"),
        # the pressure by the zero-padded FFT convolution
        _grid("cylinder_2048_fft", "fft", "cylinder", 2048, 12, 0.75, 16, 0.0, 0),
        # forces and moments from volume sums alone (the cross-check of the surface forces)
        _grid("cylinder_2048_volume_forces", "forces", "cylinder", 2048, 12, 0.75, 16, 0.0, 0),
        # an adaptive grid refined towards the body: mixed precision, and FP64 with surface points
        _adaptive("adaptive_mixed", 3, 8, 12, 0.5, 0, "mixed"),
        _adaptive("adaptive_fp64_surface", 3, 8, 20, 0.5, 2048, "fp64"),
    ]


def _grid(name, mode, flow, n, order, theta, tile, theta_surface, npts, precision="mixed", interp="nearest"):
    return {"name": name, "mode": mode, "flow": flow, "n": n, "order": order, "theta": theta, "tile": tile,
            "theta_surface": theta_surface, "npts": npts, "precision": precision, "interp": interp}


def _adaptive(name, lmin, lmax, order, theta, npts, precision, cx=0.3, cy=0.5, radius=0.05):
    return {"name": name, "mode": "adaptive", "lmin": lmin, "lmax": lmax, "order": order, "theta": theta,
            "npts": npts, "precision": precision, "cx": cx, "cy": cy, "radius": radius}


def draw(rng):
    """One more case: the modes above over the sizes, orders, acceptances and tiles in use."""
    def family(c):
        return (c["mode"] == "adaptive", c["precision"])
    while True:
        c = _draw_any(rng)
        if _cost(c) <= max(_cost(x) for x in listed() if family(x) == family(c)):
            return c


def _draw_any(rng):
    order = rng.choice([12, 12, 16, 20])
    theta = rng.choice([0.4, 0.5, 0.6, 0.7, 0.75])
    npts = int(round(math.exp(rng.uniform(math.log(256), math.log(8192)))))
    mode = rng.choice(["graph", "graph", "calls", "fp64", "fft", "forces", "batch", "adaptive", "adaptive"])
    if mode == "adaptive":
        precision = rng.choice(["mixed", "fp64"])
        c = _adaptive("", rng.choice([2, 3, 4]), rng.choice([5, 6, 7, 8]), rng.choice([8, 12, 16, 20]),
                      rng.choice([0.5, 0.6, 0.75]), npts if precision == "fp64" else 0, precision,
                      round(rng.uniform(0.25, 0.75), 3), round(rng.uniform(0.25, 0.75), 3),
                      round(rng.uniform(0.02, 0.1), 3))
    elif mode == "batch":
        c = {"mode": "batch", "flow": "swimmer", "count": rng.randint(2, 16), "nmin": rng.choice([128, 256]),
             "nmax": rng.choice([512, 1024, 2048]), "order": order, "theta": max(theta, 0.6),
             "tile": rng.choice([16, 128]), "theta_surface": rng.choice([0.0, 0.5]), "npts": npts,
             "precision": "mixed"}
    elif mode == "fp64":
        c = _grid("", "calls", rng.choice(["vortex", "cylinder", "swimmer"]), rng.choice([64, 128, 256, 512, 1024]),
                  rng.choice([12, 16, 20]), max(theta, 0.5), 16, 0.0, npts, "fp64", rng.choice(["nearest", "bilinear"]))
    elif mode == "fft":
        fp64 = rng.random() < 0.3
        c = _grid("", "fft", rng.choice(["cylinder", "swimmer"]), rng.choice([256, 512, 1024] + [2048] * (not fp64)),
                  12, 0.75, 16, 0.0, 0, "fp64" if fp64 else "mixed")
    elif mode == "forces":
        c = _grid("", "forces", rng.choice(["cylinder", "swimmer"]), rng.choice([256, 512, 1024, 2048]), 12, 0.75, 16,
                  0.0, 0, rng.choice(["mixed", "mixed", "fp64"]))
    else:
        c = _grid("", mode, rng.choice(["cylinder", "swimmer"]), rng.choice([128, 256, 512, 1024, 2048, 4096]), order,
                  theta, rng.choice([8, 16, 128, 128]), rng.choice([0.0, 0.5, 0.45, 0.4]), npts, "mixed",
                  rng.choice(["nearest", "nearest", "bilinear"]))
    c.pop("name", None)
    return c


def _cost(case):
    """Rough seconds of a pass, to keep drawn cases below the largest listed one: FP64
    operations run at a sixty-fourth of the FP32 rate."""
    w = work(case)
    return w["bytes"] / 6e12 + w["flops"] / (1e12 if case["precision"] == "fp64" else 6e13)


# ---------------------------------------------------------------------------- inputs
def _blobs(X, Y, xb, yb, gam, sigma):
    """Velocity of Gaussian vortex blobs: u_theta = gam / (2 pi r) (1 - exp(-r^2 / sigma^2))."""
    u, v = torch.zeros_like(X), torch.zeros_like(X)
    for xc, yc, g in zip(xb, yb, gam):
        dx, dy = X - float(xc), Y - float(yc)
        r2 = (dx * dx + dy * dy).clamp_(min=1e-30)
        k = torch.expm1(r2 * (-1.0 / sigma ** 2)).div_(r2).mul_(-float(g) / (2 * math.pi))
        u -= dy.mul_(k)
        v += dx.mul_(k)
    return u, v


def _heaviside(d, eps):
    t = (d / eps).clamp_(-1.0, 1.0)
    return 0.5 * (1.0 + t + torch.sin(math.pi * t) / math.pi)


def _midline(s, L, phase):
    A = 0.125 * L * (0.03125 + s / L) / 1.03125
    arg = 2 * np.pi * (s / L - phase)
    dy = 0.125 / 1.03125 * np.sin(arg) + A * (2 * np.pi / L) * np.cos(arg)
    dx = np.sqrt(np.clip(1.0 - dy * dy, 0.0, None))
    x = np.concatenate([[0.0], np.cumsum(0.5 * (dx[1:] + dx[:-1]) * np.diff(s))])
    return 0.4 + x, 0.5 + A * np.sin(arg)


def _snapshot(flow, n, npts, seed):
    """u, v, chi, us_x, us_y (float64 CUDA, n x n), points and normals (CUDA), lift, U_inf, lambda, nu."""
    rng = np.random.default_rng([seed, n])
    h = 1.0 / n
    c = (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * h
    Y, X = torch.meshgrid(c, c, indexing="ij")
    zero = torch.zeros_like(X)
    if flow == "vortex":
        xc, yc = 0.5 + 0.02 * rng.uniform(-1, 1, 2)
        u, v = _blobs(X, Y, [xc], [yc], [rng.uniform(0.5, 1.5)], 0.05)
        pts, nrm = synth.circle_surface(max(npts, 3), (xc, yc), 0.15)
        fields, lift, uinf, lam, nu = (u, v, zero, zero.clone(), zero.clone()), 0.0, (1.0, 0.0), 0.0, 0.0
    elif flow == "cylinder":
        R, (xc, yc) = 0.05, np.array([0.3, 0.5]) + 0.01 * rng.uniform(-1, 1, 2)
        dx, dy = X - xc, Y - yc
        r2 = dx * dx + dy * dy
        chi = _heaviside(R - r2.sqrt(), h)
        k = R * R / r2.clamp(min=0.25 * R * R) ** 2
        bu, bv = _blobs(X, Y, rng.uniform(xc + 0.1, 0.9, 64), rng.uniform(yc - 0.1, yc + 0.1, 64),
                        rng.normal(0.0, 0.1, 64), 2 * h)
        u = (1 - chi) * (1.0 - k * (dx * dx - dy * dy) + bu)
        v = (1 - chi) * (-2.0 * k * dx * dy + bv)
        pts, nrm = synth.circle_surface(max(npts, 3), (xc, yc), R)
        fields, lift, uinf, lam, nu = (u, v, chi, zero, zero.clone()), 2 * h, (1.0, 0.0), LAMBDA, NU
    else:
        L, phase = 0.2, rng.uniform()
        sm = np.linspace(0.0, L, 1025)
        mx, my = _midline(sm, L, phase)
        a, b = _midline(sm, L, phase + 1e-5), _midline(sm, L, phase - 1e-5)
        mid = torch.tensor(np.stack([mx, my], 1), device="cuda")
        vel = torch.tensor(np.stack([a[0] - b[0], a[1] - b[1]], 1) / 2e-5, device="cuda")
        width = torch.tensor(synth.fish_half_width(sm, L), device="cuda")
        pad = 0.05 * L + 2 * h
        i0, i1 = max(int((mx.min() - pad) * n), 0), min(int((mx.max() + pad) * n) + 1, n)
        j0, j1 = max(int((my.min() - pad) * n), 0), min(int((my.max() + pad) * n) + 1, n)
        P = torch.stack([X[j0:j1, i0:i1].reshape(-1), Y[j0:j1, i0:i1].reshape(-1)], 1)
        near = [torch.cdist(p, mid, compute_mode="donot_use_mm_for_euclid_dist").min(1) for p in P.split(1 << 16)]
        dist, at = torch.cat([m.values for m in near]), torch.cat([m.indices for m in near])
        chi, usx, usy = zero.clone(), zero.clone(), zero
        chi[j0:j1, i0:i1] = _heaviside(width[at] - dist, h).view(j1 - j0, i1 - i0)
        usx[j0:j1, i0:i1] = vel[at, 0].view(j1 - j0, i1 - i0)
        usy[j0:j1, i0:i1] = vel[at, 1].view(j1 - j0, i1 - i0)
        bu, bv = _blobs(X, Y, rng.uniform(mx[-1] + 0.05, mx[-1] + 0.35, 64), rng.uniform(0.4, 0.6, 64),
                        rng.normal(0.0, 0.1, 64), 2 * h)
        u, v = chi * usx + (1 - chi) * bu, chi * usy + (1 - chi) * bv
        half = max(npts, 4) // 2
        ss = (np.arange(half) + 0.5) * L / half
        px, py = _midline(np.concatenate([[0.0], ss]), L, phase)
        tx, ty = np.gradient(px)[1:], np.gradient(py)[1:]
        tn, ws = np.hypot(tx, ty), synth.fish_half_width(ss, L)
        ox, oy = -ty / tn * ws, tx / tn * ws
        right, left = np.stack([px[1:] - ox, py[1:] - oy], 1), np.stack([px[1:] + ox, py[1:] + oy], 1)
        pts = np.concatenate([right, left[::-1]])
        tan = np.roll(pts, -1, 0) - np.roll(pts, 1, 0)
        nrm = np.stack([tan[:, 1], -tan[:, 0]], 1)
        nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
        fields, lift, uinf, lam, nu = (u, v, chi, usx, usy), 0.0, (-1.0, 0.0), LAMBDA, NU
    return {"n": n, "h": h, "fields": fields, "pts": torch.tensor(pts, device="cuda"),
            "nrm": torch.tensor(nrm, device="cuda"), "lift": lift, "uinf": uinf, "lam": lam, "nu": nu}


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


@functools.lru_cache(maxsize=8)
def _blocks(lmin, lmax, cx, cy, radius):
    return synth.adaptive_blocks(lmin, lmax, centre=(cx, cy), radius=radius, band=2.0)


def _layout(case):
    return _blocks(case["lmin"], case["lmax"], case["cx"], case["cy"], case["radius"])


def _adaptive_inputs(case, seed):
    """Cell weights f h^2 (a smooth source around the body plus noise) and points on the body."""
    lv, ix, iy = _layout(case)
    rng = np.random.default_rng(seed)
    xs, ys, hs = synth.block_cells(lv, ix, iy)
    r = np.hypot(xs - case["cx"], ys - case["cy"]) / case["radius"]
    f = (rng.normal(size=xs.size) + 2.0 * np.exp(-r * r) + 0.5 * np.sin(2 * np.pi * xs + rng.uniform(0, 6)))
    q = torch.tensor(f * hs ** 2, device="cuda").to(_dtype(case))
    pts = synth.circle_surface(max(case["npts"], 3), (case["cx"], case["cy"]), case["radius"])[0]
    return xs, ys, hs, q, torch.tensor(pts, device="cuda")


def _snapshots(case, seed):
    if case["mode"] != "batch":
        return [_snapshot(case["flow"], case["n"], case["npts"], seed)]
    return [_snapshot(case["flow"], n, case["npts"], 1000 * seed + k) for k, n in enumerate(_batch_sizes(case))]


def _batch_sizes(case):
    sizes = [case["nmin"]]
    while sizes[-1] < case["nmax"]:
        sizes.append(2 * sizes[-1])
    return [sizes[k % len(sizes)] for k in range(case["count"])]


# ---------------------------------------------------------------------------- a pass
class _Step:
    """A snapshot in the plan's precision, its plan and output buffers."""

    def __init__(self, case, snap):
        dt = _dtype(case)
        n, npts = snap["n"], len(snap["pts"])
        self.snap = snap
        self.fields = [a.to(dt).contiguous() for a in snap.pop("fields")]
        self.plan = api.Plan(n, snap["h"], case["order"], case["theta"], precision=case["precision"],
                             lift=snap["lift"], interp=case.get("interp", "nearest"), uinf=snap["uinf"],
                             tile=case["tile"], theta_surface=case["theta_surface"])
        self.P = torch.empty(n * n, dtype=dt, device="cuda")
        self.f = torch.empty(n * n, dtype=dt, device="cuda") if case["mode"] == "calls" else None
        self.per = torch.empty(5 * npts, dtype=torch.float64, device="cuda")
        self.forces = torch.zeros(6, dtype=torch.float64, device="cuda")
        self.volume = torch.zeros(4, dtype=torch.float64, device="cuda")
        self.moments = torch.zeros(3, dtype=torch.float64, device="cuda")

    def capture(self):
        s = self.snap
        return self.plan.capture_step(*self.fields, s["lam"], p_out=self.P, points=s["pts"], normals=s["nrm"],
                                      nu=s["nu"], per_point=self.per, forces=self.forces)

    def results(self):
        return {"P": self.P, "per_point": self.per, "forces": self.forces}


def prepare(case, seed):
    if case["mode"] == "adaptive":
        _, _, _, q, pts = _adaptive_inputs(case, seed)
        return {"case": case, "tree": api.AdaptiveTree(*_layout(case), theta=case["theta"]), "q": q, "pts": pts,
                "P": torch.empty_like(q), "Ps": torch.empty(len(pts), dtype=torch.float64, device="cuda")}
    steps = [_Step(case, s) for s in _snapshots(case, seed)]
    state = {"case": case, "steps": steps}
    if case["mode"] in ("graph", "batch"):
        state["graphs"] = [s.capture() for s in steps]
    if case["mode"] == "batch":
        state["batch"] = api.Batch(state["graphs"])
    return state


def run(state):
    mode, case = state["case"]["mode"], state["case"]
    if mode == "adaptive":
        tree = state["tree"]
        if case["precision"] == "mixed":
            tree.solve_mixed(state["q"], case["order"], state["P"])
            return {"P": state["P"]}
        tree.solve(state["q"], case["order"], state["P"])
        tree.surface_pressure(state["q"], state["pts"], 0.5, state["Ps"])
        return {"P": state["P"], "P_surface": state["Ps"]}
    if mode == "batch":
        state["batch"].launch()
        return [s.results() for s in state["steps"]]
    s = state["steps"][0]
    if mode == "graph":
        state["graphs"][0].launch()
        return s.results()
    lam = s.snap["lam"]
    if mode == "forces":
        s.plan.penal_force(*s.fields, lam, forces=s.volume)
        s.plan.body_moments(*s.fields[:3], out=s.moments)
        return {"penal": s.volume, "moments": s.moments}
    if mode == "fft":
        s.plan.rhs(*s.fields, lam)
        s.plan.pressure_solve_fft(s.P)
        return {"P": s.P}
    s.plan.rhs(*s.fields, lam, f_out=s.f)
    s.plan.pressure_solve(s.P)
    s.plan.surface_traction(s.fields[0], s.fields[1], s.snap["pts"], s.snap["nrm"], s.snap["nu"], per_point=s.per,
                            forces=s.forces)
    return {"f": s.f, **s.results()}


# ---------------------------------------------------------------------------- work
def _shift(p):
    return 12 * p + 2 * p * (p + 1)


def _translation(p):
    return 16 * p + p * (4 * p + 2)


def _grid_work(case, n, npts):
    """Fields in, pressure (and source) and per-point results out; stencil, expansions, near field."""
    size, p = (8 if case["precision"] == "fp64" else 4), case["order"]
    cells = n * n
    out = {"fft": 1, "calls": 2, "forces": 0}.get(case["mode"], 1)
    if case["mode"] == "forces":
        return {"bytes": 5.0 * cells * size, "flops": 14.0 * cells}
    w = {"bytes": (5.0 + out) * cells * size, "flops": 30.0 * cells}
    if case["mode"] == "fft":
        w["flops"] += (3 * n + 2) * 5.0 * 2 * n * math.log2(2 * n) + 6.0 * 4 * cells
        return w
    w["bytes"] += npts * 9 * 8.0
    near = len(api.pp_near_offsets(case["theta"]))
    lists = sum(len(api.pp_m2l_entries(case["theta"], c)) for c in range(4)) / 4
    boxes = (cells / 64) * 4 / 3
    w["flops"] += cells * (2.0 * 64 * near + 4 * p + 8 * p) + boxes * (lists * _translation(p) + 2 * _shift(p))
    w["flops"] += npts * (250 * 8.0 * p / 8 + 9 * 64 * 10)
    return w


@functools.lru_cache(maxsize=8)
def _adaptive_pairs(lmin, lmax, cx, cy, radius, theta):
    t = api.adaptive_tree(*_blocks(lmin, lmax, cx, cy, radius), theta)
    return len(t["p2p"]), len(t["m2l"]), len(t["level"])


def work(case):
    if case["mode"] == "adaptive":
        lv, p = _layout(case)[0], case["order"]
        size, cells = (8 if case["precision"] == "fp64" else 4), len(lv) * 64
        near, far, boxes = _adaptive_pairs(case["lmin"], case["lmax"], case["cx"], case["cy"], case["radius"],
                                           case["theta"])
        return {"bytes": 2.0 * cells * size + 24.0 * case["npts"],
                "flops": 2.0 * 4096 * near + far * _translation(p) + 2.0 * boxes * _shift(p) + 12.0 * p * cells
                + case["npts"] * (150 * 8.0 * p + 9 * 64 * 30)}
    sizes = _batch_sizes(case) if case["mode"] == "batch" else [case["n"]]
    parts = [_grid_work(case, n, case["npts"]) for n in sizes]
    return {k: sum(w[k] for w in parts) for k in ("bytes", "flops")}


# ---------------------------------------------------------------------------- 64-bit results
def _source64(u, v, chi, usx, usy, h, lam):
    def d(a, axis):
        g = torch.gradient(a, spacing=h, dim=axis, edge_order=2)[0]
        return g
    f = -(d(u, 1) ** 2 + 2 * d(u, 0) * d(v, 1) + d(v, 0) ** 2)
    return f + lam * (d(chi * (usx - u), 1) + d(chi * (usy - v), 0)) if lam else f


def _grid_sum64(q, n, h):
    """(1/2 pi) sum q log max(r, rho_h) at every cell, by a zero-padded FFT convolution."""
    i = torch.arange(2 * n, device="cuda", dtype=torch.float64)
    i = torch.minimum(i, 2 * n - i)
    r2 = (i[:, None] ** 2 + i[None, :] ** 2).clamp_(min=RHO_H ** 2)
    kernel = torch.fft.rfft2(r2.log_().mul_(0.5).add_(math.log(h)).div_(2 * math.pi))
    return torch.fft.irfft2(kernel.mul_(torch.fft.rfft2(q, s=(2 * n, 2 * n))), s=(2 * n, 2 * n))[:n, :n].contiguous()


def _point_sum64(q, x, y, rho, pts):
    """The same sum at points, over cells (x, y) whose distance is clamped at rho."""
    out = torch.zeros(len(pts), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 27) // len(pts))
    for k in range(0, len(q), step):
        r2 = (pts[:, :1] - x[None, k:k + step]) ** 2
        r2 += (pts[:, 1:] - y[None, k:k + step]) ** 2
        r2 = torch.maximum(r2, rho[None, k:k + step] ** 2)
        out += r2.log_() @ q[k:k + step]
    return out * (0.5 / (2 * math.pi))


def _traction64(u, v, s, P, interp):
    n, h, pts, nrm = s["n"], s["h"], s["pts"], s["nrm"]

    def grad(i, j):
        return ((u[j, i + 1] - u[j, i - 1]) / (2 * h), (u[j + 1, i] - u[j - 1, i]) / (2 * h),
                (v[j, i + 1] - v[j, i - 1]) / (2 * h), (v[j + 1, i] - v[j - 1, i]) / (2 * h))
    at = (pts + s["lift"] * nrm) / h
    if interp == "nearest":
        c = at.floor().long().clamp(1, n - 2)
        g = grad(c[:, 0], c[:, 1])
    else:
        at = at - 0.5
        c = at.floor().long().clamp(1, n - 3)
        a = (at - c).clamp(0.0, 1.0)
        g = [0.0] * 4
        for k in range(4):
            w = (a[:, 0] if k & 1 else 1 - a[:, 0]) * (a[:, 1] if k >> 1 else 1 - a[:, 1])
            g = [x + w * y for x, y in zip(g, grad(c[:, 0] + (k & 1), c[:, 1] + (k >> 1)))]
    dxy, mu2 = 0.5 * (g[1] + g[2]), 2.0 * s["nu"]
    t_nu = torch.stack([mu2 * (g[0] * nrm[:, 0] + dxy * nrm[:, 1]), mu2 * (dxy * nrm[:, 0] + g[3] * nrm[:, 1])], 1)
    t_p = -P[:, None] * nrm
    length = (pts.roll(-1, 0) - pts).norm(dim=1)
    dS = 0.5 * (length + length.roll(1, 0))
    Fp, Fn = (t_p * dS[:, None]).sum(0), (t_nu * dS[:, None]).sum(0)
    F, (ux, uy) = Fp + Fn, s["uinf"]
    per = torch.cat([P[:, None], t_p, t_nu], 1).reshape(-1)
    return per, torch.stack([*Fp, *Fn, F[0] * ux + F[1] * uy, -F[0] * uy + F[1] * ux])


def _exact_step(case, s):
    n, h = s["n"], s["h"]
    u, v, chi, usx, usy = [a.to(_dtype(case)).double() for a in s.pop("fields")]
    if case["mode"] == "forces":
        F = s["lam"] * h * h * torch.stack([(chi * (u - usx)).sum(), (chi * (v - usy)).sum()])
        ux, uy = s["uinf"]
        return {"penal": torch.stack([*F, F[0] * ux + F[1] * uy, -F[0] * uy + F[1] * ux]),
                "moments": torch.stack([h * h * chi.sum(), (chi * u).sum() / chi.sum(), (chi * v).sum() / chi.sum()])}
    f = _source64(u, v, chi, usx, usy, h, s["lam"])
    del chi, usx, usy
    q = f * h * h
    out = {"P": _grid_sum64(q, n, h).view(-1)}
    if case["mode"] == "fft":
        return out
    c = (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * h
    x, y = c.repeat(n), c.repeat_interleave(n)
    Ps = _point_sum64(q.view(-1), x, y, torch.full_like(x, RHO_H * h), s["pts"])
    out["per_point"], out["forces"] = _traction64(u, v, s, Ps, case.get("interp", "nearest"))
    if case["mode"] == "calls":
        out = {"f": f.view(-1), **out}
    return out


def exact(case, seed):
    if case["mode"] == "adaptive":
        xs, ys, hs, q, pts = _adaptive_inputs(case, seed)
        x, y, rho = (torch.tensor(a, device="cuda") for a in (xs, ys, RHO_H * hs))
        q = q.double()
        cells = torch.stack([x, y], 1)
        out = {"P": torch.cat([_point_sum64(q, x, y, rho, c) for c in cells.split(8192)])}
        if case["precision"] == "fp64":
            out["P_surface"] = _point_sum64(q, x, y, rho, pts)
        return out
    if case["mode"] != "forces" and sum(n * n for n in (_batch_sizes(case) if case["mode"] == "batch" else [case["n"]])
                                        ) * case["npts"] > 1.2e11:
        return None
    steps = [_exact_step(case, s) for s in _snapshots(case, seed)]
    return steps if case["mode"] == "batch" else steps[0]
