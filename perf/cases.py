"""Timed workloads of the forward semi-Lagrangian library, through its public Python entry points.

Every case is one call (or one advance of a batch) that a user's program makes over and over: a step
of the paper's test flows, a plain remap, a shallow-water or Burgers step, a batch of small grids, a
served job.  `listed()` holds the representative sizes, `draw()` more of the same ranges, `prepare()`
what the program holds before the call, `run()` the call, `work()` the bytes and operations the call
cannot do without, and `exact()` the same result from plain FP64 torch, written here from the method's
definition.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1410_2817_gb300 import inputs, sl

DEV = "cuda"
SL_TYPE = {"f32": sl.SL_F32, "f64": sl.SL_F64}
TORCH_TYPE = {"f32": torch.float32, "f64": torch.float64}


# ------------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------------
def _case(name, kind, n, fields, dtype, **kw):
    c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2] if len(n) > 2 else 1, "fields": fields, "dtype": dtype,
         "order": 1, "steps": 1}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: the paper's solid-body rotation of a cone and a slotted disk, a quarter
        # turn in 16 steps of one FP64 field, where launches and latency count
        _case("sbr64_f64", "sbr", (64, 64), 1, "f64", steps=16),
        # the headline: one production step of the swirling deformation flow, three fields; the
        # program's time advances from call to call
        _case("swirl1024_f32", "swirl", (1024, 1024), 3, "f32"),
        # the same step in FP64, for runs that compare with the double-precision oracle
        _case("swirl1024_f64", "swirl", (1024, 1024), 3, "f64"),
        # a remap alone, for a program that moves the nodes itself
        _case("remap1024_f32", "remap", (1024, 1024), 3, "f32"),
        # the quintic spline (order 2 with drops to 1 and 0) on the headline flow
        _case("quintic1024_f32", "swirl", (1024, 1024), 3, "f32", order=2),
        # 2-D Burgers, whose velocity is carried by the fields: four steps per call
        _case("burgers1024_f32", "burgers", (1024, 1024), 2, "f32", steps=4),
        # the nonlinear Kelvin wave with viscosity: shallow-water stages and the quintic remap
        _case("kelvin512_f32", "kelvin", (512, 512), 3, "f32", order=2, steps=2),
        # a served 2-D job: random Fourier velocity, odd rows, four fields
        _case("job2d_723_f32", "job", (723, 723), 4, "f32"),
        # 512 independent grids of sides 32 to 512, two fields each, advanced together by the time
        # step the server gives its batched jobs
        _case("batch512_f32", "batch", (32, 512), 2, "f32", count=512),
        # the large call: the 3-D deformation flow on 256^3, two fields
        _case("deform256_f32", "deform", (256, 256, 256), 2, "f32"),
        # served 3-D jobs: an odd side in FP32 with three fields, and the FP64 option
        _case("job3d_79_f32", "job", (79, 79, 79), 3, "f32"),
        _case("job3d_64_f64", "job", (64, 64, 64), 2, "f64"),
    ]


def draw(rng):
    def side(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["sbr", "swirl", "swirl", "swirl64", "remap", "remap", "quintic", "burgers", "kelvin", "job2d",
                       "job2d", "job2d64", "batch", "deform", "job3d", "job3d", "job3d64"])
    if kind == "sbr":
        n = side(48, 160)
        return _case(None, "sbr", (n, n), 1, "f64", steps=rng.choice([8, 16]))
    if kind in ("swirl", "remap"):
        return _case(None, kind, (side(128, 2048), side(128, 2048)), rng.randint(1, 4), "f32")
    if kind == "swirl64":
        return _case(None, "swirl", (side(64, 1024), side(64, 1024)), rng.randint(1, 3), "f64")
    if kind == "quintic":
        return _case(None, "swirl", (side(128, 1536), side(128, 1536)), rng.randint(1, 4), "f32", order=2)
    if kind == "burgers":
        n = side(384, 1536)
        return _case(None, "burgers", (n, n), 2, "f32", steps=rng.choice([1, 2, 4]))
    if kind == "kelvin":
        n = side(128, 1024)
        return _case(None, "kelvin", (n, n), 3, "f32", order=2, steps=rng.choice([1, 2]))
    if kind in ("job2d", "job2d64"):
        n = side(64, 2048 if kind == "job2d" else 1024)
        return _case(None, "job", (n, n), rng.randint(1, 4), "f32" if kind == "job2d" else "f64")
    if kind == "batch":
        return _case(None, "batch", (32, 512), 2, "f32", count=rng.choice([64, 96, 128, 200, 256, 384]))
    if kind == "deform":
        n = side(64, 224)
        return _case(None, "deform", (n, n, n), rng.randint(1, 2), "f32")
    n = side(32, 192 if kind == "job3d" else 72)
    return _case(None, "job", (n, n, n), rng.randint(1, 4), "f32" if kind == "job3d" else "f64")


def _dim(case):
    return 3 if case["nz"] > 1 else 2


def _sides(case):
    return (case["nx"], case["ny"], case["nz"])[: _dim(case)]


def _batch_sides(case):
    rng = np.random.default_rng([case["count"], 7])
    lo, hi = math.log(case["nx"]), math.log(case["ny"])
    return [int(v) for v in np.round(np.exp(rng.uniform(lo, hi, size=case["count"])))]


# ------------------------------------------------------------------------------------------------
# inputs: velocity, time step and fields, from the case and the seed alone
# ------------------------------------------------------------------------------------------------
def _coords(n, lo):
    """FP64 node coordinates of a lattice on the unit-length box from lo, one plane per axis (x
    first), shaped (nz,) ny, nx."""
    ax = [lo[a] + torch.arange(n[a], device=DEV, dtype=torch.float64) / n[a] for a in range(len(n))]
    return list(reversed(torch.meshgrid(*reversed(ax), indexing="ij")))


def _near(d):
    return d - torch.round(d)


def _gauss(x, c, sigma):
    return torch.exp(-sum(_near(xa - ca) ** 2 for xa, ca in zip(x, c)) / (2 * sigma * sigma))


def _ball(x, c, r):
    return (sum(_near(xa - ca) ** 2 for xa, ca in zip(x, c)) < r * r).double()


def _setup(case, seed):
    """(velocity kind, its parameters, dt, t0, box lo, FP64 fields) of a single-grid case."""
    rng = np.random.default_rng([seed, 3])
    n, dim, kind = _sides(case), _dim(case), case["kind"]
    lo = (0.0, -0.5) if kind == "kelvin" else (0.0,) * dim
    x = _coords(n, lo)
    t0 = 0.0
    if kind == "sbr":  # cone and slotted disk, jittered about the paper-like positions
        cx, cy, dx, dy = rng.uniform(-0.03, 0.03, size=4) + np.array([0.5, 0.75, 0.5, 0.25])
        cone = torch.clamp(1.0 - torch.hypot(x[0] - cx, x[1] - cy) / 0.15, min=0.0)
        slot = (torch.abs(x[0] - dx) <= 0.025) & (x[1] <= dy + 0.1)
        disk = (torch.hypot(x[0] - dx, x[1] - dy) <= 0.15) & ~slot
        return "solid_body", [2 * math.pi, 0.5, 0.5], 1.0 / n[0], t0, lo, torch.stack([cone + disk.double()])
    if kind in ("swirl", "remap"):
        t0 = float(rng.uniform(0.0, 1.5))
        c = rng.uniform(0.3, 0.7, size=(case["fields"], 2))
        planes = []
        for f in range(case["fields"]):
            if f % 3 == 0:
                planes.append(_gauss(x, c[f], 0.1))
            elif f % 3 == 1:
                planes.append(_ball(x, c[f], 0.2))
            else:
                planes.append(torch.sin(2 * math.pi * (x[0] - c[f, 0])) * torch.sin(2 * math.pi * (x[1] - c[f, 1])))
        return "swirl2d", [5.0], 5.0 / max(n), t0, lo, torch.stack(planes)
    if kind == "burgers":  # the paper's radial pulse
        cx, cy = rng.uniform(0.45, 0.55, size=2)
        rx, ry = x[0] - cx, x[1] - cy
        r = torch.hypot(rx, ry)
        amp = torch.where(r > 0.001, torch.exp(-150.0 * (r - 0.2) ** 2) / torch.clamp(r, min=0.001), torch.zeros_like(r))
        return "carried", [], 0.5 / n[0], t0, lo, torch.stack([amp * rx, amp * ry])
    if kind == "kelvin":  # amplitude 0.5, nu 0.0005, CFL 0.5
        s = _near(x[0] - float(rng.uniform(0.0, 1.0)))
        h = 0.5 * torch.exp(-125.0 * x[1] ** 2) * torch.exp(-125.0 * s ** 2)
        return "nlsw", [250.0, 0.0005], 0.5 / n[0], t0, lo, torch.stack([h, h, torch.zeros_like(h)])
    if kind == "deform":
        t0 = float(rng.uniform(0.0, 1.0))
        c = rng.uniform(0.33, 0.67, size=(2, 3))
        planes = [_gauss(x, c[0], 0.08), _ball(x, c[1], 0.15)][: case["fields"]]
        return "deform3d", [3.0], 7.68 / n[0], t0, lo, torch.stack(planes)
    # a served job: random divergence-free Fourier velocity, alternating Gaussians and balls
    p = inputs.fourier2d_params(rng) if dim == 2 else inputs.fourier3d_params(rng)
    dt = 4.0 / (n[0] * inputs.fourier_speed_bound(p, dim))
    c = rng.uniform(0.2, 0.8, size=(case["fields"], dim))
    planes = [_gauss(x, c[f], 0.1) if f % 2 == 0 else _ball(x, c[f], 0.15) for f in range(case["fields"])]
    return ("fourier2d" if dim == 2 else "fourier3d"), p, dt, t0, lo, torch.stack(planes)


def _batch_setup(case, seed):
    """Per grid: side, Fourier parameters, dt; and one flat FP32 buffer with every grid's planes
    (each grid's planes start on a 512-byte boundary)."""
    rng = np.random.default_rng([seed, 5])
    grids, size = [], 0
    for n in _batch_sides(case):
        grids.append({"n": n, "p": inputs.fourier2d_params(rng), "at": size, "c": rng.uniform(0.25, 0.75, size=(2, 2))})
        size += -(-case["fields"] * n * n // 128) * 128
    flat = torch.zeros(size, device=DEV)
    for g in grids:
        n = g["n"]
        x = _coords((n, n), (0.0, 0.0))
        flat[g["at"]: g["at"] + 2 * n * n] = torch.stack([_gauss(x, g["c"][0], 0.1), _ball(x, g["c"][1], 0.2)]).float().reshape(-1)
        g["dt"] = 4.0 / (n * inputs.fourier_speed_bound(g["p"], 2))
    return grids, flat


def prepare(case, seed):
    if case["kind"] == "batch":
        grids, flat = _batch_setup(case, seed)
        work, scratch = flat.clone(), torch.zeros_like(flat)
        handles = [sl.Grid(2, (g["n"], g["n"]), 2, sl.SL_F32, velocity="fourier2d", velocity_params=g["p"]) for g in grids]

        def planes(buf):
            return [buf[g["at"]: g["at"] + 2 * g["n"] ** 2].view(2, g["n"], g["n"]) for g in grids]

        batch = sl.Batch(handles, planes(work), planes(scratch), [0.0] * len(grids), [g["dt"] for g in grids])
        return {"kind": "batch", "batch": batch, "first": flat, "work": work, "scratch": scratch, "grids": handles}
    vel, params, dt, t0, lo, fields = _setup(case, seed)
    n, dim = _sides(case), _dim(case)
    hi = tuple(v + 1.0 for v in lo)
    threshold = -1.0 if vel == "nlsw" else 0.25
    g = sl.Grid(dim, n, case["fields"], SL_TYPE[case["dtype"]], lo=lo, hi=hi, max_order=case["order"],
                limiter_threshold=threshold, velocity=vel, velocity_params=params)
    fin = fields.to(TORCH_TYPE[case["dtype"]])
    state = {"kind": case["kind"], "grid": g, "in": fin, "out": torch.empty_like(fin), "dt": dt, "t": t0,
             "steps": case["steps"]}
    state["scratch"] = torch.empty_like(fin) if case["steps"] > 1 or vel == "nlsw" else None
    if case["kind"] == "remap":
        g.advect(t0, dt)
    return state


def run(state):
    if state["kind"] == "batch":
        # every pass advances the ensemble from its initial fields
        state["work"].copy_(state["first"])
        state["batch"].step(1, use_graph=False)
        return state["work"]
    g = state["grid"]
    if state["kind"] == "remap":
        g.remap(state["in"], state["out"])
        return state["out"]
    g.step_out(state["in"], state["out"], state["t"], state["dt"], state["steps"], state["scratch"])
    state["t"] += state["steps"] * state["dt"]
    return state["out"]


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without: every field read and written once per step (and the displacement
# read by a plain remap); the multiplications and additions of the trajectories, the element
# inversion, the jump tests and the spline sums per node
# ------------------------------------------------------------------------------------------------
def work(case):
    dim, F, size = _dim(case), case["fields"], 8 if case["dtype"] == "f64" else 4
    taps = (2 * case["order"] + 2) ** dim
    flops = (60 if dim == 2 else 260) + F * (2 * taps + 8 * dim)
    if case["kind"] == "batch":
        nodes = sum(n * n for n in _batch_sides(case))
        return {"bytes": 2.0 * F * size * nodes, "flops": float(flops * nodes)}
    nodes = float(np.prod(_sides(case)))
    if case["kind"] == "remap":
        return {"bytes": (2 * F + dim) * size * nodes, "flops": flops * nodes}
    flops += {"swirl": 150, "deform": 300, "kelvin": 500, "burgers": 2}.get(case["kind"], 0)
    return {"bytes": 2.0 * F * size * nodes, "flops": float(flops * nodes * case["steps"])}


# ------------------------------------------------------------------------------------------------
# the same results in plain FP64 torch, from the method's definition
# ------------------------------------------------------------------------------------------------
class _Lattice:
    """Nodes of one periodic lattice, or of several 2-D lattices one after another (then the sides
    and the first node are tensors with a value per node)."""

    def __init__(self, n, base=0):
        self.n, self.base, self.dim = n, base, len(n)

    def at(self, which):
        def pick(v):
            return v[which] if torch.is_tensor(v) else v
        return _Lattice([pick(v) for v in self.n], pick(self.base))

    def index(self, k):
        i = torch.remainder(k[-1], self.n[-1])
        for a in range(self.dim - 2, -1, -1):
            i = i * self.n[a] + torch.remainder(k[a], self.n[a])
        return i + self.base


def _corner(v, dim):
    return [(v >> a) & 1 for a in range(dim)]


def _solve(J, r):
    """J x = r by cofactors, J[a][b] = d x_a / d xi_b; returns (det, x)."""
    if len(r) == 2:
        det = J[0][0] * J[1][1] - J[0][1] * J[1][0]
        return det, [(r[0] * J[1][1] - J[0][1] * r[1]) / det, (J[0][0] * r[1] - r[0] * J[1][0]) / det]

    def det3(c0, c1, c2):
        return (c0[0] * (c1[1] * c2[2] - c1[2] * c2[1]) - c1[0] * (c0[1] * c2[2] - c0[2] * c2[1])
                + c2[0] * (c0[1] * c1[2] - c0[2] * c1[1]))

    c = [[J[a][b] for a in range(3)] for b in range(3)]
    det = det3(*c)
    return det, [det3(r, c[1], c[2]) / det, det3(c[0], r, c[2]) / det, det3(c[0], c[1], r) / det]


def _invert(P, dim):
    """Newton inversion of the multilinear map with vertices P[v][a] relative to the target:
    local coordinates and 0 (converged), 1 (iteration cap) or 2 (folded element)."""
    A = [[P[1 << b][a] - P[0][a] for b in range(dim)] for a in range(dim)]
    det, x = _solve(A, [-P[0][a] for a in range(dim)])
    x = torch.stack(x)
    status = torch.where(det > 0, 1, 2)
    x[:, status == 2] = math.nan
    todo = torch.nonzero(status == 1)[:, 0]
    for _ in range(8):
        if todo.numel() == 0:
            break
        s = [x[a, todo] for a in range(dim)]
        F = [torch.zeros_like(s[0]) for _ in range(dim)]
        J = [[torch.zeros_like(s[0]) for _ in range(dim)] for _ in range(dim)]
        for v in range(1 << dim):
            o = _corner(v, dim)
            w = [s[a] if o[a] else 1 - s[a] for a in range(dim)]
            for a in range(dim):
                p = P[v][a][todo]
                F[a] = F[a] + math.prod(w) * p
                for b in range(dim):
                    J[a][b] = J[a][b] + (1 if o[b] else -1) * math.prod([w[q] for q in range(dim) if q != b]) * p
        det, d = _solve(J, F)
        fold = ~(det > 0)
        d = torch.where(fold, 0.0, torch.stack(d))
        x[:, todo] -= d
        status[todo[fold]] = 2
        done = ~fold & (d.abs().amax(0) <= 1e-14)
        status[todo[done]] = 0
        todo = todo[~fold & ~done]
    return x, status


def _locate(lat, D, j):
    """Element search: (cell, local coordinates, found) of the targets j."""
    dim = lat.dim
    Dj = D[:, lat.index(j)]
    c = torch.stack([torch.floor(j[a] - Dj[a]).long() for a in range(dim)])
    x = torch.zeros_like(Dj)
    found = torch.zeros_like(c[0], dtype=torch.bool)
    todo = torch.arange(c.shape[1], device=DEV)
    for _ in range(64):
        if todo.numel() == 0:
            break
        part, ct = lat.at(todo), c[:, todo]
        P = []
        for v in range(1 << dim):
            o = _corner(v, dim)
            k = [ct[a] + o[a] for a in range(dim)]
            i = part.index(k)
            P.append([(k[a] - j[a][todo]).double() + D[a, i] for a in range(dim)])
        xi, status = _invert(P, dim)
        x[:, todo] = xi
        finite = torch.isfinite(xi).all(0)
        low, high = xi < -1e-12, xi > 1 + 1e-12
        inside = finite & ~(low | high).any(0)
        found[todo[inside & (status == 0)]] = True
        on = finite & ~inside
        todo = todo[on]
        c[:, todo] += high[:, on].long() - low[:, on].long()
    return c, x, found


def _spline(m, x):
    """Cardinal Z-splines of order 0, 1, 2 at |x| = a."""
    a = x.abs()
    if m == 0:
        return torch.clamp(1 - a, min=0.0)
    if m == 1:
        w = torch.where(a <= 1, 1 - 2.5 * a ** 2 + 1.5 * a ** 3, 0.5 * (2 - a) ** 2 * (1 - a))
        return torch.where(a <= 2, w, 0.0)
    s, u = a - 1, 3 - a
    inner = 1 + a * a * (-1.25 + a * (-35 / 12 + a * (5.25 - a * 25 / 12)))
    middle = s * (-2 / 3 + s * (2 / 3 + s * (1.625 + s * (-8 / 3 + s * 25 / 24))))
    outer = u ** 3 * (7 / 24 + u * (-0.5 + u * 5 / 24))
    return torch.where(a <= 1, inner, torch.where(a <= 2, middle, torch.where(a <= 3, outer, 0.0)))


def _remap(lat, j, D, h, order, threshold, chunk=1 << 22):
    """One remap of the planes h (F, nodes) with the displacement D (dim, nodes) in cell units."""
    dim, N = lat.dim, h.shape[1]

    def moved(f, a, o):  # the planes' values at node + o along axis a
        return f[:, lat.index([j[b] + (o if b == a else 0) for b in range(dim)])]

    jump = torch.zeros_like(h, dtype=torch.bool)
    if threshold >= 0:
        for a in range(dim):
            up, down = moved(h, a, 1) - h, h - moved(h, a, -1)
            jump |= (up - down).abs() > threshold * torch.maximum(up.abs(), down.abs())
    boxes = {}
    for m in range(1, order + 1):  # any jump in the stencil c-m .. c+m+1 of element c
        b = jump
        for a in range(dim):
            b = torch.stack([moved(b, a, o) for o in range(-m, m + 2)]).any(0)
        boxes[m] = b
    out = torch.empty_like(h)
    for at in range(0, N, chunk):
        sel = torch.arange(at, min(N, at + chunk), device=DEV)
        part, jt = lat.at(sel), [v[sel] for v in j]
        c, x, found = _locate(part, D, jt)
        ci = part.index(list(c))
        m_of = torch.full((h.shape[0], sel.numel()), order, device=DEV)
        for m in range(order, 0, -1):
            m_of = torch.where((m_of == m) & boxes[m][:, ci], m - 1, m_of)
        val = h[:, sel].clone()
        for m in range(order + 1):
            taps = range(-m, m + 2)
            w = [[_spline(m, x[a] - t) for t in taps] for a in range(dim)]
            acc = torch.zeros_like(val)
            for kz in (range(len(taps)) if dim == 3 else (0,)):
                for ky in range(len(taps)):
                    for kx in range(len(taps)):
                        k = [c[0] + taps[kx], c[1] + taps[ky]] + ([c[2] + taps[kz]] if dim == 3 else [])
                        wt = w[0][kx] * w[1][ky] * (w[2][kz] if dim == 3 else 1.0)
                        acc += wt * h[:, part.index(k)]
            val = torch.where((m_of == m) & found, acc, val)
        out[:, sel] = val
    return out


def _velocity(kind, p, x, t):
    pi = math.pi
    if kind == "solid_body":
        return [p[0] * (p[2] - x[1]), p[0] * (x[0] - p[1])]
    if kind == "swirl2d":
        ct = math.cos(pi * t / p[0])
        return [torch.sin(pi * x[0]) ** 2 * torch.sin(2 * pi * x[1]) * ct,
                -torch.sin(pi * x[1]) ** 2 * torch.sin(2 * pi * x[0]) * ct]
    if kind == "deform3d":
        ct = math.cos(pi * t / p[0])
        s, d = [torch.sin(pi * v) ** 2 for v in x], [torch.sin(2 * pi * v) for v in x]
        return [2 * s[0] * d[1] * d[2] * ct, -s[1] * d[2] * d[0] * ct, -s[2] * d[0] * d[1] * ct]
    dim = len(x)
    u = [torch.zeros_like(x[0]) for _ in range(dim)]
    for m in p:  # Fourier modes: (kx, ky, a, b) of a streamfunction, (k, a, b) of a vector potential
        th = 2 * pi * sum(m[a] * x[a] for a in range(dim))
        s, c = torch.sin(th), torch.cos(th)
        if dim == 2:
            d = 2 * pi * (m[3] * c - m[2] * s)
            u = [u[0] + m[1] * d, u[1] - m[0] * d]
        else:
            q = [2 * pi * (c * m[6 + a] - s * m[3 + a]) for a in range(3)]
            u = [u[a] + m[(a + 1) % 3] * q[(a + 2) % 3] - m[(a + 2) % 3] * q[(a + 1) % 3] for a in range(3)]
    return u


def _advect(kind, p, X, t, dt):
    """Classical RK4 displacement over [t, t + dt], physical units."""
    def at(u, s):
        return [xa + s * ua for xa, ua in zip(X, u)]

    k1 = _velocity(kind, p, X, t)
    k2 = _velocity(kind, p, at(k1, dt / 2), t + dt / 2)
    k3 = _velocity(kind, p, at(k2, dt / 2), t + dt / 2)
    k4 = _velocity(kind, p, at(k3, dt), t + dt)
    return torch.stack([dt / 6 * (a + 2 * b + 2 * c + d) for a, b, c, d in zip(k1, k2, k3, k4)])


def _shallow_water(h, n, lo, f0, nu, dt):
    """The three low-storage RK3 stages on the nodes with fourth-order lattice differences: node
    values and displacement (cells)."""
    W = h.reshape(-1, n[1], n[0]).clone()
    q, e, eq = torch.zeros_like(W), torch.zeros_like(W[:2]), torch.zeros_like(W[:2])
    y0 = (lo[1] + torch.arange(n[1], device=DEV, dtype=torch.float64) / n[1])[:, None]

    def diff(f, a):
        d = 1 - a

        def r(o):
            return torch.roll(f, -o, dims=d)
        return (2 / 3 * (r(1) - r(-1)) - 1 / 12 * (r(2) - r(-2))) * n[a]

    for A, B in ((0.0, 1 / 3), (-5 / 9, 15 / 16), (-153 / 128, 8 / 15)):
        J = [[(1.0 if a == b else 0.0) + diff(e[a], b) for b in range(2)] for a in range(2)]
        det = J[0][0] * J[1][1] - J[0][1] * J[1][0]
        I = [[J[1][1] / det, -J[0][1] / det], [-J[1][0] / det, J[0][0] / det]]

        def grad(f):
            g = [diff(f, 0), diff(f, 1)]
            return [g[0] * I[0][b] + g[1] * I[1][b] for b in range(2)]

        gh, gu, gv = grad(W[0]), grad(W[1]), grad(W[2])
        f = f0 * (y0 + e[1])
        S = [-(1 + W[0]) * (gu[0] + gv[1]), -gh[0] + f * W[2], -gh[1] - f * W[1]]
        if nu:
            t11, t12, t22 = (1 + W[0]) * 2 * gu[0], (1 + W[0]) * (gu[1] + gv[0]), (1 + W[0]) * 2 * gv[1]
            S[1] = S[1] + nu * (grad(t11)[0] + grad(t12)[1])
            S[2] = S[2] + nu * (grad(t12)[0] + grad(t22)[1])
        q = A * q + dt * torch.stack(S)
        eq = A * eq + dt * W[1:3]
        W, e = W + B * q, e + B * eq
    cells = torch.stack([e[0] * n[0], e[1] * n[1]])
    return W.reshape(h.shape), cells.reshape(2, -1)


def exact(case, seed):
    if case["kind"] == "batch":
        grids, flat = _batch_setup(case, seed)
        sides = torch.tensor([g["n"] for g in grids], device=DEV)
        first = torch.cumsum(sides * sides, 0) - sides * sides
        of = torch.repeat_interleave(torch.arange(len(grids), device=DEV), sides * sides)
        n, base = sides[of], first[of]
        local = torch.arange(of.numel(), device=DEV) - base
        j = [local % n, local // n]
        at = torch.tensor([g["at"] for g in grids], device=DEV)[of]
        places = torch.stack([at + local, at + n * n + local])
        p = torch.tensor([g["p"][1:] for g in grids], device=DEV, dtype=torch.float64).reshape(len(grids), -1, 4)[of]
        dt = torch.tensor([g["dt"] for g in grids], device=DEV, dtype=torch.float64)[of]
        modes = [[p[:, q, k] for k in range(4)] for q in range(p.shape[1])]
        X = [v.double() / n for v in j]
        D = _advect("fourier2d", modes, X, 0.0, dt) * n
        out = torch.zeros(flat.numel(), device=DEV, dtype=torch.float64)
        out[places] = _remap(_Lattice([n, n], base), j, D, flat.double()[places], 1, 0.25)
        return out
    vel, p, dt, t0, lo, fields = _setup(case, seed)
    n, dim = _sides(case), _dim(case)
    h = fields.to(TORCH_TYPE[case["dtype"]]).double()
    shape, h = h.shape, h.reshape(h.shape[0], -1)
    i = torch.arange(h.shape[1], device=DEV)
    j = [i % n[0], (i // n[0]) % n[1], i // (n[0] * n[1])][:dim]
    X = [lo[a] + j[a].double() / n[a] for a in range(dim)]
    cells = torch.tensor(n, device=DEV, dtype=torch.float64)[:, None]
    if vel.startswith("fourier"):
        p = [p[1 + k: 1 + k + (4 if dim == 2 else 9)] for k in range(0, len(p) - 1, 4 if dim == 2 else 9)]
    lat = _Lattice(list(n))
    for s in range(case["steps"]):
        if vel == "nlsw":
            h, D = _shallow_water(h, n, lo, p[0], p[1], dt)
        elif vel == "carried":
            D = dt * h[:2] * cells
        else:
            D = _advect(vel, p, X, t0 + s * dt, dt) * cells
        h = _remap(lat, j, D, h, case["order"], -1.0 if vel == "nlsw" else 0.25)
    return h.reshape(shape)
