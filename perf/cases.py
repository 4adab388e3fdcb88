"""Performance cases of the library, through its public entry points.

Twelve named cases (`listed`), a generator of further ones over the same
ranges (`draw`), and for each case its inputs (`prepare`), one pass (`run`),
the work no implementation can do without (`work`) and the same outputs from
plain torch in binary64 (`exact`), written from the equations of arXiv
1311.3004 with none of the library's code.

A simulation case holds a solver in mid-run: a pass advances it by a chunk of
time steps and reads the state out, as a program does that watches its run.
"""
import math
import random

import numpy as np
import torch
import torch.nn.functional as F

from paper_1311_3004_gb300 import fvna

PERIODIC, EXTRAP, REFLECT, TAYLOR, HIFU = 0, 1, 2, 3, 4
BETA, DELTA = 3.5, 4.3e-6 / (1500.0 * 1.5e-3)   # water at 1 MHz
TISSUE_BETA, TISSUE_DELTA, TISSUE_AMP = 4.8, 2.974e-4, 4.217e-4
RATIO = 1e-7                                    # Taylor shock: diffusivity over beta


def listed():
    return [
        # plane-wave shock formation, 512x8: the smallest run, where latency and launches count
        {"name": "plane_512x8_f64", "kind": "plane", "bits": 64, "nx": 512, "ny": 8, "steps": 32},
        # the 2D Gaussian pulse at its configured size, in both precisions
        {"name": "pulse_2048_f64", "kind": "pulse", "bits": 64, "nx": 2048, "ny": 2048, "steps": 8},
        {"name": "pulse_2048_f32", "kind": "pulse", "bits": 32, "nx": 2048, "ny": 2048, "steps": 32},
        # the driven axisymmetric focused source at its configured size
        {"name": "focused_4096x1024_f32", "kind": "focused", "bits": 32, "nx": 4096, "ny": 1024,
         "steps": 16},
        # the focused packet study (28 x 20 wavelengths, 20 cells each): the axis is read after
        # every step, so each step is a call of its own
        {"name": "packet_560x400_f64", "kind": "packet", "bits": 64, "nx": 560, "ny": 400,
         "steps": 8},
        # the rotated Taylor shock on its moving 100-unit window, 10 cells per unit
        {"name": "taylor_1000_f64", "kind": "taylor", "bits": 64, "nx": 1000, "ny": 1000,
         "steps": 32},
        # many independent domains of uneven size in one context
        {"name": "batch_48_f32", "kind": "batch", "bits": 32, "domains": 48, "smallest": 256,
         "largest": 1536, "sizes": 4, "steps": 16},
        # a small ragged domain with Strang steps
        {"name": "strang_257x129_f32", "kind": "strang", "bits": 32, "nx": 257, "ny": 129,
         "steps": 32},
        # 3D: a ragged box in binary64, the configured 256^3 pulse in binary32
        {"name": "box_145x130x113_f64", "kind": "box", "bits": 64, "nx": 145, "ny": 130, "nz": 113,
         "steps": 4},
        {"name": "box_256_f32", "kind": "box", "bits": 32, "nx": 256, "ny": 256, "nz": 256,
         "steps": 8},
        # the correction network on one coarse 2048x512 field, and one step of its training on
        # eight 128x128 crops
        {"name": "net_forward_2048x512", "kind": "forward", "batch": 1, "h": 512, "w": 2048},
        {"name": "net_train_8x128x128", "kind": "train", "batch": 8, "h": 128, "w": 128},
    ]


def _size(rng, lo, hi):
    """A whole size spread over the logarithm of its range."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["plane", "pulse", "pulse", "focused", "packet", "taylor", "batch",
                       "strang", "box", "box", "forward", "train"])
    bits = rng.choice([32, 64])
    if kind == "plane":
        return {"kind": kind, "bits": bits, "nx": _size(rng, 64, 2048), "ny": _size(rng, 4, 40),
                "steps": rng.choice([16, 32])}
    if kind == "pulse":
        return {"kind": kind, "bits": bits, "nx": _size(rng, 48, 2000), "ny": _size(rng, 48, 2000),
                "steps": 8 if bits == 64 else 24}
    if kind == "focused":
        return {"kind": kind, "bits": bits, "nx": _size(rng, 256, 3900 if bits == 32 else 2048),
                "ny": _size(rng, 64, 1000 if bits == 32 else 512), "steps": 8}
    if kind == "packet":
        return {"kind": kind, "bits": bits, "nx": _size(rng, 200, 1100), "ny": _size(rng, 100, 800),
                "steps": rng.choice([4, 8])}
    if kind == "taylor":
        n = _size(rng, 100, 1000)
        return {"kind": kind, "bits": 64, "nx": n, "ny": n, "steps": 16}
    if kind == "batch":
        return {"kind": kind, "bits": 32, "domains": rng.randint(4, 32), "smallest": 200,
                "largest": rng.randint(300, 1400), "sizes": rng.randint(0, 999), "steps": 16}
    if kind == "strang":
        return {"kind": kind, "bits": bits, "nx": _size(rng, 33, 700), "ny": _size(rng, 33, 500),
                "steps": 16}
    if kind == "box":
        top = 240 if bits == 32 else 120
        return {"kind": kind, "bits": bits, "nx": _size(rng, 24, top), "ny": _size(rng, 24, top),
                "nz": _size(rng, 24, top), "steps": 4}
    if kind == "forward":
        return {"kind": kind, "batch": rng.choice([1, 1, 2]), "h": _size(rng, 64, 512),
                "w": _size(rng, 64, 1024)}
    return {"kind": kind, "batch": rng.randint(2, 8), "h": _size(rng, 32, 128),
            "w": _size(rng, 32, 128)}


# ---------------------------------------------------------------- inputs

def _grid(nx, ny, dx, x0=0.0, y0=0.0):
    x = x0 + (torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5) * dx
    y = y0 + (torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5) * dx
    return x[None, :], y[:, None]


def _at_rest(*shape):
    q = torch.zeros((len(shape) + 1,) + shape, device="cuda", dtype=torch.float64)
    q[0] = 1.0
    return q


def _domains(case, seed):
    """(run parameters, [(domain parameters, state)]) of a 2D case."""
    r = random.Random(seed)
    kind = case["kind"]
    p = {"beta": BETA, "delta": DELTA, "dx": 1.0 / 40.0, "nu": 0.9, "axisymmetric": False,
         "strang": kind == "strang"}
    d = {"bc": (EXTRAP,) * 4, "x0": 0.0, "y0": 0.0, "t0": 0.0, "ratio": 0.0, "angle": 0.0,
         "amp": 0.0, "focal": 1.0, "aperture": 0.0, "envelope": 0}
    if kind == "batch":
        sizes = random.Random(case["sizes"])
        out = []
        for _ in range(case["domains"]):
            n = sizes.randint(case["smallest"], case["largest"])
            amp = math.exp(r.uniform(math.log(0.1e6), math.log(2.0e6))) / 2.25e9
            f, ang = r.uniform(0.5, 2.0), r.uniform(0.0, 2.0 * math.pi)
            X, Y = _grid(n, n, f * p["dx"])
            c, s, mid = math.cos(ang), math.sin(ang), 0.5 * n * f * p["dx"]
            xi = (X - mid) * c + (Y - mid) * s
            w = amp * torch.sin(2 * math.pi * xi) * torch.exp(-(xi / 2.0) ** 2)
            q = _at_rest(n, n)
            q[0] += w
            q[1], q[2] = w * c, w * s
            out.append((dict(d, nx=n, ny=n), q))
        return p, out
    nx, ny = case["nx"], case["ny"]
    d["nx"], d["ny"] = nx, ny
    q = _at_rest(ny, nx)
    if kind == "plane":          # a 1 MPa sine along x1
        d["bc"] = (EXTRAP, EXTRAP, PERIODIC, PERIODIC)
        X, _ = _grid(nx, ny, p["dx"])
        w = 1.0e6 / 2.25e9 * r.uniform(0.8, 1.2) * torch.sin(2 * math.pi * (X + r.random()))
        q[0] += w
        q[1] += w
    elif kind == "pulse":        # a 2 MPa Gaussian at rest, sigma 8 cells
        X, Y = _grid(nx, ny, 1.0)
        cx, cy = nx * r.uniform(0.4, 0.6), ny * r.uniform(0.4, 0.6)
        q[0] += 2.0e6 / 2.25e9 * torch.exp(-((X - cx) ** 2 + (Y - cy) ** 2) / 128.0)
    elif kind == "strang":       # a few smooth modes in all fields
        d["bc"] = (PERIODIC, PERIODIC, REFLECT, EXTRAP)
        p["delta"] = 1e-3
        X, Y = _grid(nx, ny, 1.0)
        for k in range(3):
            for _ in range(4):
                q[k] += 2.5e-4 * r.uniform(-1, 1) * torch.cos(
                    2 * math.pi * (r.randint(0, 3) * X / nx + r.randint(0, 3) * Y / ny
                                   + r.random()))
    elif kind == "focused":      # the driven beam some periods after its start
        p["dx"], p["nu"], p["axisymmetric"] = 1.0 / 30.0, 0.4, True
        d.update(bc=(HIFU, EXTRAP, REFLECT, EXTRAP), amp=0.3e6 / 2.25e9 * r.uniform(0.8, 1.2),
                 focal=40.0, aperture=min(20.0, 0.6 * ny / 30.0), t0=30.0 + r.random())
        X, Y = _grid(nx, ny, p["dx"])
        tau = d["t0"] + Y * Y / (2.0 * d["focal"]) - X
        e = torch.where(tau > 0, torch.exp(-(tau.clamp(min=1e-3) / 4.0) ** -10), 0.0 * tau)
        w = d["amp"] * torch.sin(2 * math.pi * tau) * e * torch.exp(-(Y / d["aperture"]) ** 8)
        q[0] += w
        q[1] += w
        q[2] -= w * Y / d["focal"]
    elif kind == "packet":       # soft tissue, the packet half way in
        p.update(beta=TISSUE_BETA, delta=TISSUE_DELTA, dx=1.0 / 20.0)
        d.update(bc=(HIFU, EXTRAP, REFLECT, EXTRAP), amp=TISSUE_AMP * r.uniform(0.8, 1.2),
                 focal=50.0, aperture=0.5 * ny / 20.0, envelope=1, t0=1.0 + r.random())
        X, Y = _grid(nx, ny, p["dx"])
        tau = d["t0"] + Y * Y / (2.0 * d["focal"]) - X
        w = d["amp"] * torch.sin(2 * math.pi * tau) * torch.exp(-(tau / 4.0) ** 10)
        w = w * torch.exp(-(Y / d["aperture"]) ** 8)
        q[0] += w
        q[1] += w
        q[2] -= w * Y / d["focal"]
    elif kind == "taylor":       # the analytic profile, centred in the window
        p.update(delta=RATIO * BETA, dx=1.0 / 10.0)
        half = 0.5 * nx * p["dx"]
        d.update(bc=(TAYLOR,) * 4, x0=-half + 0.1 * r.random(), y0=-half + 0.1 * r.random(),
                 ratio=RATIO, angle=math.pi / 8)
        X, Y = _grid(nx, ny, p["dx"], d["x0"], d["y0"])
        c, s = math.cos(d["angle"]), math.sin(d["angle"])
        w = -RATIO * torch.tanh(X * c + Y * s)
        q[0] += w
        q[1], q[2] = w * c, w * s
    return p, [(d, q)]


def _box(case, seed):
    r = random.Random(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    a = [torch.arange(n, device="cuda", dtype=torch.float64) + 0.5 - n * r.uniform(0.4, 0.6)
         for n in (nx, ny, nz)]
    q = _at_rest(nz, ny, nx)
    r2 = a[0][None, None, :] ** 2 + a[1][None, :, None] ** 2 + a[2][:, None, None] ** 2
    q[0] += 2.0e6 / 2.25e9 * torch.exp(-r2 / 128.0)
    return q


def _net(case, seed):
    g = torch.Generator().manual_seed(seed)
    rng = np.random.default_rng(seed)
    flat = []
    for o, c in ((32, 3), (32, 32), (3, 32)):
        std = math.sqrt(2.0 / (9 * c)) * (0.1 if o == 3 else 1.0)
        flat.append(rng.normal(0.0, std, size=9 * o * c))
        flat.append(rng.normal(0.0, 0.01, size=o))
    shape = (case["batch"], 3, case["h"], case["w"])
    x = torch.randn(shape, generator=g).cuda()
    t = torch.randn(shape, generator=g).cuda() if case["kind"] == "train" else None
    return np.concatenate(flat).astype(np.float32), x, t


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("forward", "train"):
        flat, x, t = _net(case, seed)
        return {"kind": kind, "net": fvna.Net(flat), "x": x, "t": t}
    prec = fvna.FP64 if case["bits"] == 64 else fvna.FP32_PERT
    s = {"kind": kind, "steps": case["steps"]}
    if kind == "box":
        q = _box(case, seed)
        cfg = fvna.make_config(precision=prec, beta=BETA, delta=DELTA, dx=1.0 / 40.0, nu_w=0.9,
                               steps_per_graph=case["steps"])
        dom = fvna.make_domain3(case["nx"], case["ny"], case["nz"])
        return dict(s, solver=fvna.Solver3(cfg, dom, q), out=[torch.empty_like(q)])
    p, doms = _domains(case, seed)
    cfg = fvna.make_config(
        precision=prec, geometry=fvna.AXISYMMETRIC if p["axisymmetric"] else fvna.CARTESIAN,
        beta=p["beta"], delta=p["delta"], dx=p["dx"], nu_w=p["nu"],
        splitting=fvna.SPLIT_STRANG if p["strang"] else fvna.SPLIT_GODUNOV,
        steps_per_graph=1 if kind == "packet" else case["steps"])
    ds = [fvna.make_domain(d["nx"], d["ny"], bc=d["bc"], envelope=d["envelope"], x0=d["x0"],
                           y0=d["y0"], t0=d["t0"], taylor_ratio=d["ratio"],
                           taylor_angle=d["angle"], amp=d["amp"], focal=d["focal"],
                           aperture=d["aperture"]) for d, _ in doms]
    solver = fvna.Solver(cfg, ds, [q for _, q in doms])
    return dict(s, solver=solver, out=[torch.empty_like(q) for _, q in doms],
                angle=doms[0][0]["angle"])


# ---------------------------------------------------------------- one pass

def run(state):
    kind = state["kind"]
    if kind == "forward":
        return state["net"].forward(state["x"])
    if kind == "train":
        loss = state["net"].train_step(state["x"], state["t"], 5e-4, margin=4)
        return {"loss": loss, "params": state["net"].params()}
    s = state["solver"]
    if kind == "packet":
        axis = []
        for _ in range(state["steps"]):
            s.run(max_steps=1)
            axis.append(s.axis_pressure(0))
        return {"axis_q1": 1.0 + np.stack(axis), "q": s.q(0, out=state["out"][0])}
    if kind == "taylor":
        a = state["angle"]
        s.run_moving(math.inf, 0.0, (math.cos(a), math.sin(a)), every=state["steps"],
                     max_steps=state["steps"])
        return [s.q(0, out=state["out"][0]), np.array(s.corner(0))]
    s.run(max_steps=state["steps"])
    if kind == "box":
        return s.q(out=state["out"][0])
    return [s.q(k, out=o) for k, o in enumerate(state["out"])]


# ---------------------------------------------------------------- what a pass cannot do without

def work(case):
    kind = case["kind"]
    if kind in ("forward", "train"):
        pix = case["batch"] * case["h"] * case["w"]
        macs = 9 * (3 * 32 + 32 * 32 + 32 * 3) * pix
        if kind == "forward":
            return {"bytes": 24 * pix, "flops": 2 * macs}
        # forward, weight gradients of all layers, input gradients of the last two
        return {"bytes": 24 * pix, "flops": 2 * (2 * macs + 9 * (32 * 32 + 32 * 3) * pix)}
    # The time step needs the largest speed of the whole field, so each step reads the state and
    # writes it; a pass then writes it once more in binary64.  Operations per cell and step, each
    # add, multiply, divide and root counted once: a 2D sweep 178, its source 19; a 3D sweep 234,
    # its source 39.  Strang steps have a third sweep.
    esz, steps = case["bits"] // 8, case["steps"]
    if kind == "batch":
        sizes = random.Random(case["sizes"])
        cells = sum(sizes.randint(case["smallest"], case["largest"]) ** 2
                    for _ in range(case["domains"]))
    else:
        cells = case["nx"] * case["ny"] * case.get("nz", 1)
    fields = 4 if kind == "box" else 3
    ops = 3 * 234 + 39 if kind == "box" else (3 if kind == "strang" else 2) * 178 + 19
    return {"bytes": cells * fields * (2 * esz * steps + 8), "flops": cells * steps * ops}


# ---------------------------------------------------------------- the same in plain binary64

def _ghosts(u, dim, n, rules, values=(None, None)):
    """The line ends of a tuple of fields: two ghost cells on each side of dimension `dim`, by
    the border rule of each side; u[1] is the normal momentum.  values: (mask, fields) of a
    driven side, with the nearest ghost last on the low side and first on the high side."""
    out = []
    for k, a in enumerate(u):
        parts = []
        for side in (0, 1):
            near = [0, 1] if side == 0 else [n - 1, n - 2]
            if rules[side] == PERIODIC:
                pick = [n - 1, n - 2] if side == 0 else [0, 1]
            elif rules[side] == REFLECT:
                pick = near
            else:
                pick = [near[0], near[0]]
            g = [a.narrow(dim, i, 1) for i in pick]
            if rules[side] == REFLECT and k == 1:
                g = [-x for x in g]
            g = torch.cat(g[::-1] if side == 0 else g, dim)
            if values[side] is not None:
                mask, v = values[side]
                g = torch.where(mask, v[k], g)
            parts.append(g)
        out.append(torch.cat([parts[0], a, parts[1]], dim))
    return out


def _waves(u, beta, dim):
    """Speeds and waves of every interface of the padded line fields u (q1, normal, transverse)."""
    n = u[0].shape[dim]
    L = [a.narrow(dim, 0, n - 1) for a in u]
    R = [a.narrow(dim, 1, n - 1) for a in u]
    Z1 = 0.5 * (L[0] + R[0])
    Z = [0.5 * (a / L[0] + b / R[0]) for a, b in zip(L[1:], R[1:])]
    vel = [z / Z1 for z in Z]
    speed = vel[0]
    c = torch.sqrt(speed * speed - 2 * Z[0] * speed + 1 + 2 * (beta - 1) * (Z1 - 1))
    s1, s2 = speed + c, speed - c
    d = [b - a for a, b in zip(L, R)]
    a1 = (d[1] - s2 * d[0]) / (2 * c)
    a2 = (s1 * d[0] - d[1]) / (2 * c)
    r1 = [v * (s1 - 2 * Z[0]) / c for v in vel[1:]]
    r2 = [v * (2 * Z[0] - s2) / c for v in vel[1:]]
    zero = torch.zeros_like(a1)
    fam = [(s1, [a1, a1 * s1] + [a1 * x for x in r1]), (s2, [a2, a2 * s2] + [a2 * x for x in r2])]
    for k, dk in enumerate(d[2:]):
        w = [zero] * len(u)
        w[2 + k] = dk - a1 * r1[k] - a2 * r2[k]
        fam.append((speed, w))
    return fam


def _sweep(u, dim, beta, lam, first_order=0):
    """One sweep of the padded fields u; returns the updated cells and max |s| over their faces.
    first_order: faces at the low end that take no correction."""
    m = u[0].shape[dim]
    n = m - 4
    fam = _waves(u, beta, dim)
    k = len(u)
    am, ap, Fl = [0.0] * k, [0.0] * k, [0.0] * k
    smax = 0.0
    for s, W in fam:
        mid = [w.narrow(dim, 1, n + 1) for w in W]
        sm = s.narrow(dim, 1, n + 1)
        smax = max(smax, float(sm.abs().max()))
        up = sm > 0
        ww, wu = 0.0, 0.0
        for w, x in zip(W, mid):
            ww = ww + x * x
            wu = wu + x * torch.where(up, w.narrow(dim, 0, n + 1), w.narrow(dim, 2, n + 1))
        theta = wu / torch.where(ww > 0, ww, torch.ones_like(ww))
        phi = torch.minimum((1 + theta) / 2, 2 * theta).clamp(0.0, 2.0)
        phi = torch.where(ww > 0, phi, torch.zeros_like(phi))
        if first_order:
            phi.narrow(dim, 0, first_order).zero_()
        a = sm.abs()
        coef = 0.5 * a * (1 - lam * a) * phi
        for i, x in enumerate(mid):
            am[i] = am[i] + sm.clamp(max=0.0) * x
            ap[i] = ap[i] + sm.clamp(min=0.0) * x
            Fl[i] = Fl[i] + coef * x
    new = []
    for i in range(k):
        q = u[i].narrow(dim, 2, n)
        new.append(q - lam * (am[i].narrow(dim, 1, n) + ap[i].narrow(dim, 0, n))
                   - lam * (Fl[i].narrow(dim, 1, n) - Fl[i].narrow(dim, 0, n)))
    return new, smax


def _taylor(d, x, y, t):
    c, s = math.cos(d["angle"]), math.sin(d["angle"])
    w = -d["ratio"] * torch.tanh(x * c + y * s - t)
    return [1.0 + w, w * c, w * s]


def _driven2(d, p, side, t):
    """(mask, (q1, q2, q3)) of the two ghost layers of a driven side, or None."""
    rule, dx = d["bc"][side], p["dx"]
    n = d["nx"] if side < 2 else d["ny"]
    at = torch.tensor([-2.0, -1.0] if side % 2 == 0 else [n, n + 1.0], device="cuda",
                      dtype=torch.float64) + 0.5
    if rule == TAYLOR:
        x, y = _grid(d["nx"], d["ny"], dx, d["x0"], d["y0"])
        x, y = (d["x0"] + at[None, :] * dx, y) if side < 2 else (x, d["y0"] + at[:, None] * dx)
        v = _taylor(d, x, y, t)
        return torch.ones_like(v[0], dtype=torch.bool), v
    if rule == HIFU and side == 0:
        _, y = _grid(d["nx"], d["ny"], dx, d["x0"], d["y0"])
        x = d["x0"] + at[None, :] * dx
        tau = t + y * y / (2 * d["focal"]) - x
        if d["envelope"] == 0:
            e = torch.where(tau > 0, torch.exp(-1.0 / (tau.clamp(min=1e-3) / 4) ** 10), 0.0 * tau)
        else:
            e = torch.exp(-(tau / 4) ** 10)
        g = d["amp"] * torch.sin(2 * math.pi * tau) * e
        rn = torch.sqrt(y * y + d["focal"] ** 2)
        return (y <= d["aperture"]) & (x < 0), [1.0 + g, d["focal"] * g / rn, -y * g / rn]
    return None


def _pad2(q, d, p, dim, t):
    """q = (q1, q2, q3) padded along dim (1: x1, 0: x2), in the sweep's order."""
    if dim == 1:
        v = tuple(_driven2(d, p, s, t) for s in (0, 1))
        return _ghosts(list(q), 1, d["nx"], d["bc"][:2], v)
    v = []
    for s in (2, 3):
        g = _driven2(d, p, s, t)
        v.append(None if g is None else (g[0], [g[1][0], g[1][2], g[1][1]]))
    return _ghosts([q[0], q[2], q[1]], 0, d["ny"], d["bc"][2:], tuple(v))


def _laplace_ends(z, dim):
    n = z.shape[dim]
    return z.narrow(dim, 0, n - 2), z.narrow(dim, 2, n - 2)


def _source2(q, d, p, dt, t):
    ux = [a.narrow(1, 1, d["nx"] + 2) for a in _pad2(q, d, p, 1, t)]
    uy = [a.narrow(0, 1, d["ny"] + 2) for a in _pad2(q, d, p, 0, t)]
    dx = p["dx"]
    coef = dt * p["delta"] / dx ** 2
    z = [q[1] / q[0], q[2] / q[0]]
    new = [q[0], None, None]
    _, y = _grid(d["nx"], d["ny"], dx, d["x0"], d["y0"])
    for k, (ix, iy) in enumerate(((1, 2), (2, 1))):
        w, e = _laplace_ends(ux[ix] / ux[0], 1)
        s, n = _laplace_ends(uy[iy] / uy[0], 0)
        lap = w + e + s + n - 4 * z[k]
        if p["axisymmetric"]:
            lap = lap + (n - s) * (dx / (2 * y))
            if k == 1:
                lap = lap - z[1] * (dx * dx / (y * y))
        new[k + 1] = q[k + 1] + coef * lap
    if p["axisymmetric"]:
        new[0] = q[0] - dt * q[2] / y
        new[1] = new[1] - dt * z[0] * z[1] / y
        new[2] = new[2] - dt * z[1] * z[1] / y
    return new


def _step2(q, d, p, t, dt):
    lam, smax = dt / p["dx"], 0.0

    def along(dim, q, lam):
        axis = 2 if p["axisymmetric"] and dim == 0 and d["y0"] == 0.0 else 0
        u, s = _sweep(_pad2(q, d, p, dim, t), dim, p["beta"], lam, axis)
        return (u if dim == 1 else [u[0], u[2], u[1]]), s

    half = 0.5 if p["strang"] else 1.0
    q, s = along(1, q, half * lam)
    smax = max(smax, s)
    q, s = along(0, q, lam)
    smax = max(smax, s)
    q = _source2(q, d, p, dt, t)
    if p["strang"]:
        q, s = along(1, q, half * lam)
        smax = max(smax, s)
    return q, smax


def _first_speed(pads, beta, dims):
    top = 0.0
    for u, dim in zip(pads, dims):
        n = u[0].shape[dim] - 4
        for s, _ in _waves(u, beta, dim)[:2]:
            top = max(top, float(s.narrow(dim, 1, n + 1).abs().max()))
    return top


def _run2(q, d, p, steps, after=None):
    q, t = list(q), d["t0"]
    dt = p["nu"] * p["dx"] / _first_speed([_pad2(q, d, p, 1, t), _pad2(q, d, p, 0, t)], p["beta"],
                                          (1, 0))
    for _ in range(steps):
        q, smax = _step2(q, d, p, t, dt)
        t += dt
        dt = p["nu"] * p["dx"] / smax
        if after:
            after(q)
    return q, t


def _moved(q, d, p, t, kx, ky):
    """The window moved by (kx, ky) cells; entering cells take the analytic profile."""
    ny, nx = q[0].shape
    d = dict(d, x0=d["x0"] + kx * p["dx"], y0=d["y0"] + ky * p["dx"])
    X, Y = _grid(nx, ny, p["dx"], d["x0"], d["y0"])
    new = _taylor(d, X, Y, t)
    ox, oy = slice(max(0, kx), nx + min(0, kx)), slice(max(0, ky), ny + min(0, ky))
    ix, iy = slice(max(0, -kx), nx + min(0, -kx)), slice(max(0, -ky), ny + min(0, -ky))
    for a, b in zip(new, q):
        a[iy, ix] = b[oy, ox]
    return new, d


def _pad3(q, dim):
    """The four fields padded along dim (2: x1, 1: x2, 0: x3), normal momentum second."""
    order = {2: (0, 1, 2, 3), 1: (0, 2, 1, 3), 0: (0, 3, 1, 2)}[dim]
    return _ghosts([q[k] for k in order], dim, q[0].shape[dim], (EXTRAP, EXTRAP))


def _run3(q, steps):
    q, dx, nu = list(q), 1.0 / 40.0, 0.9
    back = {2: (0, 1, 2, 3), 1: (0, 2, 1, 3), 0: (0, 2, 3, 1)}
    dt = nu * dx / max(_first_speed([_pad3(q, k)], BETA, (k,)) for k in (2, 1, 0))
    for _ in range(steps):
        smax = 0.0
        for dim in (2, 1, 0):
            u, s = _sweep(_pad3(q, dim), dim, BETA, dt / dx)
            q = [u[k] for k in back[dim]]
            smax = max(smax, s)
        coef = dt * DELTA / dx ** 2
        new = [q[0]]
        for k in (1, 2, 3):
            z = q[k] / q[0]
            lap = -6 * z
            for dim in (0, 1, 2):
                n = z.shape[dim]
                g = torch.cat([z.narrow(dim, 0, 1), z, z.narrow(dim, n - 1, 1)], dim)
                a, b = _laplace_ends(g, dim)
                lap = lap + a + b
            new.append(q[k] + coef * lap)
        q = new
        dt = nu * dx / smax
    return torch.stack(q)


def _exact_net(case, seed):
    flat, x, t = _net(case, seed)
    w = torch.from_numpy(flat).cuda().double().requires_grad_(case["kind"] == "train")
    at = [0]

    def take(*shape):
        n = math.prod(shape)
        at[0] += n
        return w[at[0] - n:at[0]].reshape(shape)

    h = x.double()
    for o, c in ((32, 3), (32, 32), (3, 32)):
        k = take(o, c, 3, 3)
        h = F.conv2d(h, k, take(o), padding=1)
        h = F.relu(h) if o == 32 else h
    if case["kind"] == "forward":
        return h
    loss = ((h - t.double())[:, :, 4:-4, 4:-4] ** 2).sum() / (
        case["batch"] * (case["h"] - 8) * (case["w"] - 8))
    loss.backward()
    # the first Adam step from rest, learning rate 5e-4
    g = w.grad
    return {"loss": float(loss), "params": (w - 5e-4 * g / (g.abs() + 1e-8)).detach()}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("forward", "train"):
        return _exact_net(case, seed)
    if kind == "box":
        return _run3(_box(case, seed), case["steps"])
    p, doms = _domains(case, seed)
    if kind == "packet":
        d, q = doms[0]
        axis = []
        q, _ = _run2(q, d, p, case["steps"], lambda u: axis.append(u[0][0].cpu().numpy()))
        return {"axis_q1": np.stack(axis), "q": torch.stack(q)}
    if kind == "taylor":
        d, q = doms[0]
        q, t = _run2(q, d, p, case["steps"])
        kx, ky = (math.floor(f(d["angle"]) * t / p["dx"] + 0.5) for f in (math.cos, math.sin))
        q, d = _moved(q, d, p, t, kx, ky)
        return [torch.stack(q), np.array([d["x0"], d["y0"]])]
    return [torch.stack(_run2(q, d, p, case["steps"])[0]) for d, q in doms]
