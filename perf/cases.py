"""The workloads the library's speed is measured on, as a user's program runs them.

Each case is one pass of such a program through the public entry points of
``paper_2005_04642_gb300.cmrt``: advance a lattice and read its snapshot, step
an ensemble, or take a gradient.  Sizes and parameters follow the library's own
workloads (``inputs.py``, ``bench.py``, the tests): drops of heavy fluid in a
light one, layered channels, buoyant drops between walls, the ensemble of
uneven lattices, the adjoint of the colour mismatch.  The lattices start from a
moving fluid (a vortex or a channel profile), as they do in the middle of a
run.  ``exact`` restates the method in 64 bits with plain torch operations.
"""
import math
import random

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2005_04642_gb300 import cmrt

SIDES = (64, 128, 256, 512)


def listed():
    return [
        # the static-drop study: a small lattice advanced in short runs, where launches and latency count
        dict(name="drop_64", kind="step", nx=64, ny=64, steps=100, ratio=10.0),
        # the layered channel: a strong density contrast between walls, a flat lattice
        dict(name="channel_1024x128", kind="step", nx=1024, ny=128, steps=100, ratio=100.0, walls=True, layers=True),
        # odd extents, constant shear viscosity and the ghost moment relaxed to zero
        dict(name="drops_1037x613", kind="step", nx=1037, ny=613, steps=40, ratio=10.0, eta=1.0 / 6.0, ghost=1),
        # an ordinary lattice, with its conserved quantities watched
        dict(name="drops_2048", kind="step", nx=2048, ny=2048, steps=20, ratio=10.0, watch=True),
        # the throughput workload
        dict(name="drops_8192", kind="step", nx=8192, ny=8192, steps=16, ratio=10.0),
        # buoyant drops between walls with 16-bit storage, the memory-saving forms
        dict(name="buoyant_fp16_4096x2048", kind="step", nx=4096, ny=2048, steps=20, ratio=10.0, walls=True,
             precision=2),
        dict(name="buoyant_bf16_1536x1000", kind="step", nx=1536, ny=1000, steps=40, ratio=10.0, walls=True,
             precision=1),
        # the high-order colour gradient (the paper's appendix B)
        dict(name="order6_1024x512", kind="step", nx=1024, ny=512, steps=20, ratio=8.0, order=6),
        # a parameter study: hundreds of uneven lattices in one launch per step
        dict(name="ensemble_512", kind="batch", members=512, steps=50, odd=False),
        # one iteration of a fit: objective and gradients from a fresh lattice, as an optimiser calls it
        dict(name="fit_256", kind="fit", nx=256, ny=256, steps=320, every=40),
        # gradients on a large lattice that the program keeps
        dict(name="adjoint_2048", kind="adjoint", nx=2048, ny=2048, steps=20, every=10),
        # one step's vector-Jacobian product, for an objective of the user's own
        dict(name="vjp_1024x384", kind="vjp", nx=1024, ny=384, ratio=10.0, walls=True),
    ]


def _size(rng, low, high):
    n = int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))
    return max(low, min(high, n - n % rng.choice((1, 1, 4, 32))))


def draw(rng):
    kind = rng.choice(("step", "step", "step", "step", "batch", "fit", "adjoint", "vjp"))
    if kind == "step":
        nx, ny = _size(rng, 48, 6000), _size(rng, 48, 6000)
        updates = math.exp(rng.uniform(math.log(4e5), math.log(4e8)))
        case = dict(kind=kind, nx=nx, ny=ny, steps=max(4, min(100, int(updates / (nx * ny)))),
                    ratio=round(math.exp(rng.uniform(0.0, math.log(40.0))), 3), walls=rng.random() < 0.4)
        case["precision"] = rng.choice((0, 0, 0, 1, 2))
        if case["precision"] == 0 and rng.random() < 0.2:
            case["order"] = 6
        if rng.random() < 0.25:
            case["ghost"] = 1
        if rng.random() < 0.25:
            case["eta"] = round(rng.uniform(0.1, 0.2), 4)
        return case
    if kind == "batch":
        return dict(kind=kind, members=_size(rng, 16, 384), steps=rng.randint(10, 50), odd=rng.random() < 0.5)
    if kind == "fit":
        return dict(kind=kind, nx=_size(rng, 64, 320), ny=_size(rng, 64, 320), steps=rng.randint(40, 240),
                    every=rng.choice((1, 10, 20, 40)))
    if kind == "adjoint":
        return dict(kind=kind, nx=_size(rng, 400, 2048), ny=_size(rng, 400, 2048), steps=rng.randint(8, 20),
                    every=rng.choice((1, 4, 10)))
    return dict(kind=kind, nx=_size(rng, 64, 2048), ny=_size(rng, 64, 2048), ratio=10.0, walls=rng.random() < 0.5)


# ---------------------------------------------------------------- inputs
def _params(nx, ny, ratio=10.0, walls=False, **kw):
    """Parameters for the density ratio rho0_r / rho0_b >= 1: the lighter fluid's rest fraction is 1/2."""
    p = dict(nx=nx, ny=ny, rho0_r=1.0, rho0_b=1.0 / ratio, alpha_r=1.0 - 0.5 / ratio, alpha_b=0.5, sigma=0.005,
             beta=0.67, lambda3_r=1.0, lambda3_b=1.0, lambda6=1.0, lambda7=1.0, g_acc=(0.0, 0.0), g_vol=(0.0, 0.0),
             wall_y=walls, visc_mode=0, eta=1.0 / 6.0, stencil_order=2, curvature_mode=0, fixed_K=0.0,
             ghost_N_mode=0, precision=0)
    p.update(kw)
    return p


def _drops(nx, ny, drops, periodic_y):
    """Union of tanh drops of width 2 (float32, CUDA): +1 inside, -1 outside; only each drop's box is touched."""
    out = torch.full((ny, nx), -1.0, dtype=torch.float64, device="cuda")
    for cx, cy, r in drops:
        half = int(math.ceil(r + 24.0))
        xs = np.unique(np.arange(int(cx) - half, int(cx) + half + 2) % nx)
        ys = np.arange(int(cy) - half, int(cy) + half + 2)
        ys = np.unique(ys % ny) if periodic_y else ys[(ys >= 0) & (ys < ny)]
        dx = xs - cx
        dx = dx - nx * np.round(dx / nx)
        dy = ys - cy
        if periodic_y:
            dy = dy - ny * np.round(dy / ny)
        X, Y = torch.from_numpy(dx).cuda(), torch.from_numpy(dy).cuda()
        val = torch.tanh((r - torch.sqrt(X[None, :] ** 2 + Y[:, None] ** 2)) / 2.0)
        ix = torch.from_numpy(xs).cuda()[None, :]
        iy = torch.from_numpy(ys).cuda()[:, None]
        out[iy, ix] = torch.maximum(out[iy, ix], val)
    return out.float()


def _scatter(rng, nx, ny, periodic_y):
    """One drop per 256 x 256 nodes or so (at least one), centres uniform in the box, off the nodes."""
    count = max(1, min(96, nx * ny // 65536))
    high = 0.25 * min(nx, ny) if count == 1 else min(64.0, 0.25 * min(nx, ny))
    drops = []
    for _ in range(count):
        r = rng.uniform(0.6 * high, high) if count == 1 else rng.uniform(min(10.0, 0.6 * high), high)
        cy = rng.uniform(0.0, ny) if periodic_y else rng.uniform(r + 3.0, max(r + 4.0, ny - r - 4.0))
        drops.append((rng.uniform(0.0, nx), cy, r))
    return drops


def _vortex(nx, ny, speed, seed):
    """One vortex pair across the box plus seeded noise (float32, CUDA)."""
    rng = random.Random(seed * 7 + 1)
    kx, ky = 2.0 * math.pi / nx, 2.0 * math.pi / ny
    x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :] * kx + rng.uniform(0.0, 6.0)
    y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None] * ky + rng.uniform(0.0, 6.0)
    a = speed / max(kx, ky)
    u = torch.stack([(a * ky) * torch.sin(x) * torch.cos(y), (-a * kx) * torch.cos(x) * torch.sin(y)])
    return _noisy(u, seed)


def _channel(nx, ny, speed, seed):
    """The parabolic profile between the walls plus seeded noise (float32, CUDA)."""
    s = (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) / ny
    u = torch.zeros((2, ny, nx), dtype=torch.float64, device="cuda")
    u[0] = (4.0 * speed * s * (1.0 - s))[:, None]
    return _noisy(u, seed)


def _noisy(u, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    u += 1e-4 * (2.0 * torch.rand(u.shape, generator=g, dtype=torch.float32, device="cuda") - 1.0)
    return u.float()


def _start(case, seed):
    """(params, rho_n0, u0) of a single lattice."""
    nx, ny, walls = case["nx"], case["ny"], bool(case.get("walls"))
    rng = random.Random(seed)
    p = _params(nx, ny, case.get("ratio", 10.0), walls, precision=case.get("precision", 0),
                stencil_order=case.get("order", 2), ghost_N_mode=case.get("ghost", 0))
    if "eta" in case:
        p.update(visc_mode=1, eta=case["eta"])
    if case.get("layers"):
        at = ny / 2.0 + rng.uniform(-2.0, 2.0)
        y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
        rho_n = torch.tanh((at - y) / 2.0).expand(ny, nx).float().contiguous()
        p.update(g_acc=(1e-6, 0.0))
    else:
        rho_n = _drops(nx, ny, _scatter(rng, nx, ny, not walls), not walls)
        if walls:  # light drops rising in the heavy fluid
            rho_n = -rho_n
            p.update(g_acc=(0.0, -1e-6))
    u = _channel(nx, ny, 0.02, seed) if walls else _vortex(nx, ny, 0.04, seed)
    return p, rho_n, u


def _members(case, seed):
    """The ensemble: sides drawn from SIDES (or odd ones near them), one drop each, sigma and the ratio per member."""
    rng = random.Random(seed)
    sides = [s - 7 - 2 * k for k, s in enumerate(SIDES)] if case["odd"] else SIDES
    pick = random.Random(1000 + case["members"])  # which sides: part of the case, not of the inputs
    out = []
    for k in range(case["members"]):
        n = pick.choice(sides)
        p = _params(n, n, math.exp(rng.uniform(0.0, math.log(100.0))), sigma=rng.uniform(0.001, 0.02))
        c = (n / 2.0 + rng.uniform(-3.0, 3.0), n / 2.0 + rng.uniform(-3.0, 3.0))
        out.append((p, c, n))
    return out


def _one_drop(n, c):
    x = torch.arange(n, dtype=torch.float64, device="cuda")
    d = torch.sqrt((x[None, :] - c[0]) ** 2 + (x[:, None] - c[1]) ** 2)
    return torch.tanh((n / 4.0 - d) / 2.0).float()


def _fit(case, seed):
    """Parameters, initial fields and target of a gradient: the target is a drop displaced by about a node."""
    nx, ny = case["nx"], case["ny"]
    rng = random.Random(seed)
    p = _params(nx, ny, 10.0, g_acc=(0.0, -1e-5))
    r = min(nx, ny) / 8.0 if min(nx, ny) < 400 else 48.0
    n = 1 if min(nx, ny) < 400 else max(1, nx * ny // 262144)
    drops = [(rng.uniform(0.0, nx), rng.uniform(0.0, ny), r) for _ in range(n)]
    moved = [(x + 1.0, y + 0.5, r * 1.02) for x, y, r in drops]
    return p, _drops(nx, ny, drops, True), _vortex(nx, ny, 0.02, seed), _drops(nx, ny, moved, True)


def _theta(p):
    return [p["sigma"], p["beta"], p["lambda3_r"], p["lambda3_b"], p["g_acc"][0], p["g_acc"][1]]


# ---------------------------------------------------------------- one pass
def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        with torch.no_grad():
            members = [(p, _one_drop(n, c), _vortex(n, n, 0.03, seed + k))
                       for k, (p, c, n) in enumerate(_members(case, seed))]
        return dict(case=case, batch=cmrt.Batch(members), sides=[p["nx"] for p, _, _ in members])
    if kind in ("fit", "adjoint"):
        p, rho_n, u, target = _fit(case, seed)
        state = dict(case=case, params=p, target=target, u0=u)
        if kind == "fit":
            state["theta"] = torch.tensor(_theta(p), device="cuda", requires_grad=True)
            state["rho_n0"] = rho_n.requires_grad_()
        else:
            state["lat"] = cmrt.Lattice(p, rho_n, u)
            state["start"] = torch.from_numpy(state["lat"].save()).cuda()
        return state
    p, rho_n, u = _start(case, seed)
    lat = cmrt.Lattice(p, rho_n, u)
    state = dict(case=case, lat=lat)
    if kind == "vjp":
        lat.step(4)
        state["lam"] = _lam(case, seed)
    return state


def _lam(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 5)
    return torch.randn((2, 9, case["ny"], case["nx"]), generator=g, device="cuda")


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        # a stretch of the run, then its snapshot: the fields to look at, the populations to go on from
        lat = state["lat"]
        lat.step(case["steps"])
        out = lat.fields()
        out["populations"] = lat.populations()
        if case.get("watch"):
            d = lat.diagnostics()
            out["mass"] = [d["mass_r"], d["mass_b"]]
            out["umax"] = d["umax"]
        return out
    if kind == "batch":
        batch = state["batch"]
        batch.step(case["steps"])
        fields = [batch.member(k).fields() for k in range(len(batch))]
        return {name: torch.cat([f[name].reshape(-1) for f in fields]) for name in fields[0]}
    if kind == "fit":
        theta, rho_n0 = state["theta"], state["rho_n0"]
        theta.grad = rho_n0.grad = None
        loss = cmrt.colour_mismatch(theta, rho_n0, state["params"], state["target"], case["steps"], case["every"],
                                    state["u0"])
        loss.backward()
        return {"loss": float(loss), "theta": theta.grad, "rho_n0": rho_n0.grad}
    if kind == "adjoint":
        lat = state["lat"]
        lat.load(state["start"])
        loss, grads, rho_n0 = lat.adjoint(case["steps"], state["target"], case["every"], want_rho_n0=True)
        return {"loss": loss, "theta": torch.tensor(list(grads.values())), "rho_n0": rho_n0}
    lam, grads = state["lat"].step_vjp(state["lam"])
    return {"lam": lam, "theta": torch.tensor(grads)}


def _cells(case):
    if case["kind"] == "batch":
        return sum(n * n for _, _, n in _members(case, 0))
    return case["nx"] * case["ny"]


def work(case):
    """Bytes and operations of one pass: per node and step the stored state is read once and written once (36 FP32
    populations, or twice the 64-byte 16-bit record), a reverse step reads the state and the adjoint and writes the
    adjoint; a snapshot reads the state once and writes what it returns.  About 250 FP32 operations per node and
    step, three times that for a reverse step."""
    n, kind = _cells(case), case["kind"]
    if kind == "vjp":
        return {"bytes": n * 216.0, "flops": n * 750.0}
    steps = case["steps"]
    if kind in ("fit", "adjoint"):
        return {"bytes": n * (steps * (144.0 + 216.0) + 8.0), "flops": n * steps * 1000.0}
    node = 64.0 if case.get("precision", 0) else 72.0
    out = 20.0 if kind == "batch" else 92.0
    return {"bytes": n * (steps * 2.0 * node + node + out), "flops": n * steps * 250.0}


# ---------------------------------------------------------------- the method in 64 bits
CX = (0, 1, 0, -1, -1, -1, 0, 1, 1)
CY = (0, 1, 1, 1, 0, -1, -1, -1, 0)
W = (4 / 9, 1 / 36, 1 / 9, 1 / 36, 1 / 9, 1 / 36, 1 / 9, 1 / 36, 1 / 9)
GHOST = (1, 4, -2, 4, -2, 4, -2, 4, -2)
OPPOSITE = (0, 5, 6, 7, 8, 1, 2, 3, 4)
ROWS = [[1, CX[i], CY[i], CX[i] ** 2, CY[i] ** 2, CX[i] * CY[i], GHOST[i], GHOST[i] * CX[i], GHOST[i] * CY[i]]
        for i in range(9)]  # [link][mode]
BACK = np.linalg.inv(np.array(ROWS, dtype=np.float64).T)  # [link][mode]
REACH = {2: (1.0,), 6: (4.5, -0.9, 0.1)}


def _at(a, dx, dy, walls, parity):
    """The field at (x + dx, y + dy): periodic, or mirrored with a sign beyond the walls."""
    if dx:
        a = torch.roll(a, -dx, -1)
    if not dy:
        return a
    if not walls:
        return torch.roll(a, -dy, -2)
    if dy > 0:
        return torch.cat([a[..., dy:, :], parity * torch.flip(a[..., -dy:, :], (-2,))], -2)
    return torch.cat([parity * torch.flip(a[..., :-dy, :], (-2,)), a[..., :dy, :]], -2)


def _derivative(a, axis, p, parity=1.0, order=2):
    out = 0.0
    for n, coefficient in enumerate(REACH[order], 1):
        for i in range(1, 9):
            c = (CX, CY)[axis][i]
            if c:
                out = out + (3.0 * coefficient if order == 2 else coefficient) * W[i] * c * _at(
                    a, n * CX[i], n * CY[i], p["wall_y"], parity)
    return out


def _combine(weights, fields):
    out = None
    for w, f in zip(weights, fields):
        if w:
            out = w * f if out is None else out + w * f
    return out


def _macro(R, B, p):
    """Densities, colour gradient, force and force-adjusted velocity."""
    rr, rb = sum(R), sum(B)
    rho = rr + rb
    a, b = rr / p["rho0_r"], rb / p["rho0_b"]
    rho_n = (a - b) / (a + b)
    order = p["stencil_order"]
    gx, gy = _derivative(rho_n, 0, p, order=order), _derivative(rho_n, 1, p, order=order)
    mag = gx * gx + gy * gy
    some = mag >= 1e-18
    inv = torch.where(some, torch.rsqrt(torch.where(some, mag, torch.ones_like(mag))), torch.zeros_like(mag))
    ex, ey = gx * inv, gy * inv
    K = -(_derivative(ex, 0, p) + _derivative(ey, 1, p, -1.0))
    half = 0.5 * p["sigma"]
    Gx = half * K * gx + rho * p["g_acc"][0]
    Gy = half * K * gy + rho * p["g_acc"][1]
    f = [r + b for r, b in zip(R, B)]
    ux = (_combine(CX, f) + 0.5 * Gx) / rho
    uy = (_combine(CY, f) + 0.5 * Gy) / rho
    return rr, rb, rho, rho_n, f, ex, ey, Gx, Gy, ux, uy


def _advance(R, B, p):
    """One step of the pre-collision populations (lists of nine fields per colour)."""
    rr, rb, rho, rho_n, f, ex, ey, Gx, Gy, ux, uy = _macro(R, B, p)
    order = p["stencil_order"]
    phi = 0.6 * (1.0 - p["alpha_r"]) * (rr + p["rho0_r"] / p["rho0_b"] * rb) - rho / 3.0
    Px, Py = _derivative(phi, 0, p, order=order), _derivative(phi, 1, p, order=order)
    div = _derivative(ux, 0, p, -1.0) + _derivative(uy, 1, p, -1.0)
    if p["visc_mode"] == 0:
        nr, nb = (2.0 / p["lambda3_r"] - 1.0) / 6.0, (2.0 / p["lambda3_b"] - 1.0) / 6.0
        nu = 0.5 * (nr + nb) + 0.5 * (nr - nb) * rho_n
    else:
        nu = p["eta"] / rho
    l3 = 2.0 / (6.0 * nu + 1.0)
    c = 1.0 - 0.5 * l3
    qx, qy = Gx - Px, Gy - Py
    iso = ux * Px + uy * Py - rho * div / 3.0
    S = (None, Gx, Gy, c * (2.0 * ux * qx - iso), c * (2.0 * uy * qy - iso), c * (ux * qy + uy * qx), None, None, None)
    pres = 0.6 * ((1.0 - p["alpha_r"]) * rr + (1.0 - p["alpha_b"]) * rb)
    N = 0.0 if p["ghost_N_mode"] else 1.8 * (p["alpha_r"] * rr + p["alpha_b"] * rb) - 0.8 * rho
    eq = (rho, rho * ux, rho * uy, rho * ux * ux + pres, rho * uy * uy + pres, rho * ux * uy, N, 0.0, 0.0)
    rate = (0.0, 0.0, 0.0, l3, l3, l3, p["lambda6"], p["lambda7"], p["lambda7"])
    change = []
    for m in range(9):
        if m == 0:
            change.append(None)
            continue
        d = 0.0 if m < 3 else rate[m] * (eq[m] - _combine([ROWS[i][m] for i in range(9)], f))
        change.append(d + S[m] if S[m] is not None else d)
    weight = 1.8 * ((1.0 - p["alpha_r"]) * rr + (1.0 - p["alpha_b"]) * rb) / rho
    seg = p["beta"] * rr * rb / rho * weight
    kr, kb = rr / rho, rb / rho
    outR, outB = [], []
    for i in range(9):
        g = f[i] + _combine(BACK[i][1:], change[1:])
        length = math.hypot(CX[i], CY[i])
        s = seg * (W[i] / length) * (CX[i] * ex + CY[i] * ey) if i else 0.0
        outR.append(kr * g + s)
        outB.append(kb * g - s)
    return _stream(outR, p), _stream(outB, p)


def _stream(post, p):
    """f_i(r) = P_i(r - c_i), half-way bounce-back at the walls."""
    out = []
    for i in range(9):
        a = torch.roll(post[i], CX[i], -1)
        if p["wall_y"] and CY[i]:
            back = post[OPPOSITE[i]]
            a = (torch.cat([back[..., :1, :], a[..., :-1, :]], -2) if CY[i] > 0 else
                 torch.cat([a[..., 1:, :], back[..., -1:, :]], -2))
        elif CY[i]:
            a = torch.roll(a, CY[i], -2)
        out.append(a)
    return out


def _initial(rho_n0, u, p):
    rr, rb = p["rho0_r"] * (1.0 + rho_n0) * 0.5, p["rho0_b"] * (1.0 - rho_n0) * 0.5
    rho = rr + rb
    rest = p["alpha_r"] * rr + p["alpha_b"] * rb
    moving = 1.8 * ((1.0 - p["alpha_r"]) * rr + (1.0 - p["alpha_b"]) * rb)
    ux, uy = u
    R, B = [], []
    for i in range(9):
        cu = CX[i] * ux + CY[i] * uy
        q = W[i] * rho * (3.0 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + uy * uy))
        f = (W[i] * moving if i else rest) + q
        R.append(rr / rho * f)
        B.append(rb / rho * f)
    return R, B


def _fields(R, B, p):
    rr, rb, rho, _, _, _, _, _, _, ux, uy = _macro(R, B, p)
    return {"rho_r": rr, "rho_b": rb, "ux": ux, "uy": uy,
            "p": 0.6 * ((1.0 - p["alpha_r"]) * rr + (1.0 - p["alpha_b"]) * rb)}


def _mismatch(theta, rho_n0, u, p, target, steps):
    q = dict(p, sigma=theta[0], beta=theta[1], lambda3_r=theta[2], lambda3_b=theta[3], g_acc=(theta[4], theta[5]))
    R, B = _initial(rho_n0, u, q)

    def step(*RB):
        r, b = _advance(RB[:9], RB[9:], q)
        return tuple(r) + tuple(b)

    state = tuple(R) + tuple(B)
    for _ in range(steps):
        state = checkpoint(step, *state, use_reentrant=False)
    a, b = sum(state[:9]) / p["rho0_r"], sum(state[9:]) / p["rho0_b"]
    return 0.5 * (((a - b) / (a + b) - target) ** 2).sum()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("fit", "adjoint"):
        p, rho_n, u, target = _fit(case, seed)
        value = torch.tensor(_theta(p), dtype=torch.float32 if kind == "fit" else torch.float64, device="cuda")
        theta = value.double().requires_grad_()
        rho_n = rho_n.double().requires_grad_()
        loss = _mismatch(theta, rho_n, u.double(), p, target.double(), case["steps"])
        loss.backward()
        return {"loss": float(loss), "theta": theta.grad, "rho_n0": rho_n.grad}
    if kind == "vjp":
        p, rho_n, u = _start(case, seed)
        theta = torch.tensor(_theta(p), dtype=torch.float64, device="cuda")
        with torch.no_grad():
            R, B = _initial(rho_n.double(), u.double(), p)
            for _ in range(4):
                R, B = _advance(R, B, p)
        RB = torch.stack(R + B).requires_grad_()
        theta.requires_grad_()
        q = dict(p, sigma=theta[0], beta=theta[1], lambda3_r=theta[2], lambda3_b=theta[3], g_acc=(theta[4], theta[5]))
        R, B = _advance(list(RB[:9]), list(RB[9:]), q)
        lam = _lam(case, seed).double().reshape(18, case["ny"], case["nx"])
        g = torch.autograd.grad(torch.stack(R + B), (RB, theta), lam)
        return {"lam": g[0].reshape(2, 9, case["ny"], case["nx"]), "theta": g[1]}
    with torch.no_grad():
        if kind == "batch":
            members = _members(case, seed)
            got = [None] * len(members)
            for n in sorted({m[2] for m in members}):  # the members of one side together
                ks = [k for k, m in enumerate(members) if m[2] == n]
                p = dict(members[ks[0]][0])
                for key in ("rho0_b", "alpha_r", "sigma"):
                    p[key] = torch.tensor([members[k][0][key] for k in ks], dtype=torch.float64,
                                          device="cuda")[:, None, None]
                rho_n = torch.stack([_one_drop(n, members[k][1]).double() for k in ks])
                u = torch.stack([_vortex(n, n, 0.03, seed + k).double() for k in ks], 1)
                R, B = _initial(rho_n, u, p)
                for _ in range(case["steps"]):
                    R, B = _advance(R, B, p)
                f = _fields(R, B, p)
                for at, k in enumerate(ks):
                    got[k] = {name: v[at].reshape(-1) for name, v in f.items()}
            return {name: torch.cat([g[name] for g in got]) for name in got[0]}
        p, rho_n, u = _start(case, seed)
        R, B = _initial(rho_n.double(), u.double(), p)
        del rho_n, u
        for _ in range(case["steps"]):
            R, B = _advance(R, B, p)
        out = _fields(R, B, p)
        out["populations"] = torch.stack([torch.stack(R), torch.stack(B)])
        if case.get("watch"):
            out["mass"] = [float(out["rho_r"].sum()), float(out["rho_b"].sum())]
            out["umax"] = float(torch.sqrt((out["ux"] ** 2 + out["uy"] ** 2).max()))
        return out
