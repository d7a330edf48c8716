"""The calls that this package's users make, as cases that can be timed.

One case is one pass through the public entry points: steps of a solver in each
precision and variant, a host round trip, the discrete adjoint of a step, the
gradient of a rollout, the FP64 invariants, and an ensemble of grids.  Initial
data are the repository's own workloads (vortex, pulse, shear layer,
Kelvin-Helmholtz, smooth random fields), sampled on the GPU with seeded phases
and centres.  `exact` is the same scheme in plain float64 torch: the acoustic
operator as 5 x 5 stencils on the half-cell lattice built from the paper's
monomial block, the two-Picard foot, the space-time Simpson fluxes.

The FP32 modes' states are returned as float32, the type they are computed in;
the API itself hands states out as float64 planes.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

import paper_2605_12915_gb300 as af
from paper_2605_12915_gb300.autograd import rollout

GAMMA = 1.4
CFL = 0.4


class _Grid:
    def __init__(self, nx, ny, x0, y0, h):
        self.nx, self.ny, self.x0, self.y0, self.h = nx, ny, x0, y0, h


class _Problem:
    def __init__(self, grid, gamma, state):
        self.grid, self.gamma, self.state = grid, gamma, state


def listed():
    return [
        # one step of the smallest workload with its state in host memory: a coupled
        # program that hands its state over every step; latency and launches only
        dict(name="host_vortex32_fp64", kind="host", flow="vortex", nx=32, ny=32,
             precision="fp64", variant="tai", steps=1),
        # the 32 x 32 vortex benchmark, all of its 100 steps: a run on a small grid
        dict(name="vortex32_comp", kind="step", flow="vortex", nx=32, ny=32,
             precision="fp32_comp", variant="tai", steps=100),
        # the pulse benchmark (512 x 512) in plain FP32, a stretch of 20 steps
        dict(name="pulse512_fp32", kind="step", flow="pulse", nx=512, ny=512,
             precision="fp32", variant="tai", steps=20),
        # the headline: the 2048 x 2048 shear layer with compensated averages
        dict(name="shear2048_comp", kind="step", flow="shear", nx=2048, ny=2048,
             precision="fp32_comp", variant="tai", steps=10),
        # a grid whose width is no multiple of 4, with the additive update
        dict(name="ragged333_rb_comp", kind="step", flow="smooth", nx=333, ny=250,
             precision="fp32_comp", variant="rb", steps=10),
        # the FP64 mode on the pulse workload, against which FP32 is judged
        dict(name="pulse512_fp64", kind="step", flow="pulse", nx=512, ny=512,
             precision="fp64", variant="tai", steps=5),
        # the foot-centred reference variant on a small grid
        dict(name="fc64_fp64", kind="step", flow="smooth", nx=64, ny=64,
             precision="fp64", variant="fc", steps=1),
        # one adjoint step of the Kelvin-Helmholtz gradient workload
        dict(name="adjoint_kh1024_comp", kind="adjoint", flow="kh", nx=1024, ny=1024,
             precision="fp32_comp", variant="tai", steps=1),
        # gradient through a checkpointed rollout: design loops on a mid-size grid
        dict(name="gradient_kh256_comp", kind="gradient", flow="kh", nx=256, ny=256,
             precision="fp32_comp", variant="tai", steps=20, every=8),
        # the same in FP64 (the rollout's default precision) on a small grid
        dict(name="gradient_vortex64_fp64", kind="gradient", flow="vortex", nx=64, ny=64,
             precision="fp64", variant="tai", steps=10, every=5),
        # the diagnostics of a long run
        dict(name="invariants_shear2048_comp", kind="invariants", flow="shear", nx=2048,
             ny=2048, precision="fp32_comp", variant="tai", steps=0),
        # a whole ensemble run of vortices on grids of uneven sizes: created, stepped,
        # every member's state read
        dict(name="ensemble8_fp32", kind="ensemble", flow="vortex", nx=64, ny=64, most=256,
             members=8, precision="fp32", variant="tai", steps=50),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "host", "adjoint", "gradient",
                       "invariants", "ensemble"])
    variant = rng.choice(["tai", "tai", "tai", "rb"])
    precision = rng.choice(["fp32_comp", "fp32_comp", "fp32", "fp64"])
    flow = rng.choice(["vortex", "pulse", "shear", "kh", "smooth"])
    if kind == "ensemble":
        return dict(kind=kind, flow="vortex", nx=64, ny=64, most=rng.choice([64, 128, 256]),
                    members=rng.randint(3, 16), precision=rng.choice(["fp32", "fp32_comp"]),
                    variant="tai", steps=_log_int(rng, 5, 50))
    if kind == "step" and rng.random() < 0.12:
        n = _log_int(rng, 8, 64)
        return dict(kind=kind, flow="smooth", nx=n, ny=max(8, n + rng.randint(-3, 3)),
                    precision="fp64", variant="fc", steps=1)
    most = {"step": 2048, "host": 512, "adjoint": 1024, "gradient": 256, "invariants": 2048}[kind]
    if precision == "fp64":
        most = min(most, 512 if kind in ("step", "host", "invariants") else 128)
    nx = _log_int(rng, 24, most)
    if rng.random() < 0.6:
        nx = max(24, nx // 4 * 4)  # widths that are a multiple of 4 are the usual ones
    ny = min(most, max(20, int(nx * rng.uniform(0.6, 1.5)))) if flow in ("smooth", "kh") else nx
    case = dict(kind=kind, flow=flow, nx=nx, ny=ny, precision=precision, variant=variant)
    if kind == "step":
        cells = 512 * 512 * 5 if precision == "fp64" else 2048 * 2048 * 10
        # (the additive update is only stable for a while at this time step)
        most = 20 if variant == "rb" else 100
        case["steps"] = max(1, min(_log_int(rng, 1, most), cells // (nx * ny)))
    elif kind == "host":
        case["steps"] = rng.randint(1, 3)
    elif kind == "gradient":
        case["steps"] = rng.randint(2, 20)
        case["every"] = rng.randint(1, 10)
    else:
        case["steps"] = 1 if kind == "adjoint" else 0
    return case


# ---- initial data ----------------------------------------------------------------
def _rng(seed):
    return np.random.default_rng(seed)


def _primitive(case, seed, member=0):
    """(grid, function of (x, y) tensors giving rho, u, v, p) of a workload; the
    seed moves centres and phases and adds small smooth modes."""
    r = _rng([seed, member])
    nx, ny, flow = case["nx"], case["ny"], case["flow"]
    if flow == "vortex":
        g = _Grid(nx, ny, -5.0, -5.0, 10.0 / nx)
    elif flow == "pulse":
        g = _Grid(nx, ny, -1.0, -1.0, 2.0 / nx)
    else:
        g = _Grid(nx, ny, 0.0, 0.0, 1.0 / nx)
    lx, ly = nx * g.h, ny * g.h
    ax, ay, ph = (r.uniform(0.0, 1.0) for _ in range(3))
    modes = [(k, int(r.integers(-3, 4)), int(r.integers(1, 4)), r.uniform(-1, 1),
              r.uniform(0, 2 * math.pi)) for k in range(4) for _ in range(3)]
    beta, uinf, vinf = r.uniform(3, 5), r.uniform(-1, 1), r.uniform(-1, 1)

    def wave(k, x, y):
        return sum(a * torch.cos(2 * math.pi * (mx * (x - g.x0) / lx + my * (y - g.y0) / ly) + p)
                   for kk, mx, my, a, p in modes if kk == k)

    def fn(x, y):
        if flow == "vortex":
            dx, dy = x - (2.5 * ax - 1.25), y - (2.5 * ay - 1.25)
            dx, dy = dx - lx * torch.round(dx / lx), dy - ly * torch.round(dy / ly)
            r2 = dx * dx + dy * dy
            f = beta / (2 * math.pi) * torch.exp(0.5 * (1 - r2))
            t = 1 - (GAMMA - 1) * beta ** 2 / (8 * GAMMA * math.pi ** 2) * torch.exp(1 - r2)
            rho = t ** (1 / (GAMMA - 1))
            return rho, uinf - f * dy, vinf + f * dx, rho ** GAMMA
        if flow == "pulse":
            dx, dy = x - 0.4 * (ax - 0.5), y - 0.4 * (ay - 0.5)
            rho = 1 + 0.1 * torch.exp(-(dx * dx + dy * dy) / 0.01)
            return rho, 0.02 * wave(1, x, y), 0.02 * wave(2, x, y), rho ** GAMMA
        yy = (y - g.y0) / ly
        if flow == "shear":
            u = torch.where(yy <= 0.5, torch.tanh(80 * (yy - 0.25)), torch.tanh(80 * (0.75 - yy)))
            v = 0.05 * torch.sin(2 * math.pi * (x + ph)) + 0.002 * wave(2, x, y)
            one = torch.ones_like(u + v)
            return one, u * one, v * one, one / (GAMMA * 0.01)
        if flow == "kh":
            inside = (yy - 0.5).abs() < 0.25
            z = torch.zeros_like(x * y)
            rho = torch.where(inside, 2.0, 1.0) + z
            return (rho + 2e-3 * wave(0, x, y), torch.where(inside, 0.5, -0.5) + z
                    + 2e-3 * wave(1, x, y), 0.01 * torch.sin(4 * math.pi * (x + ph)) + z
                    + 2e-3 * wave(2, x, y), 2.5 + 2e-3 * wave(3, x, y))
        return (1 + 0.05 * wave(0, x, y), 0.3 + 0.05 * wave(1, x, y),
                -0.2 + 0.05 * wave(2, x, y), (1 + 0.05 * wave(3, x, y)) / GAMMA)

    return g, fn


def _state(case, seed, member=0):
    """Grid, (16, ny, nx) float64 state on the GPU and the CFL time step: averages
    by 6 x 6 Gauss-Legendre quadrature, point values sampled."""
    g, fn = _primitive(case, seed, member)
    x = g.x0 + g.h * torch.arange(g.nx, dtype=torch.float64, device="cuda")[None, :]
    y = g.y0 + g.h * torch.arange(g.ny, dtype=torch.float64, device="cuda")[:, None]
    s = torch.empty((16, g.ny, g.nx), dtype=torch.float64, device="cuda")
    q, w = np.polynomial.legendre.leggauss(6)
    s[:4] = 0
    for a in range(6):
        for b in range(6):
            rho, u, v, p = fn(x + 0.5 * g.h * (q[a] + 1), y + 0.5 * g.h * (q[b] + 1))
            wt = 0.25 * w[a] * w[b]
            s[0] += wt * rho
            s[1] += wt * rho * u
            s[2] += wt * rho * v
            s[3] += wt * (p / (GAMMA - 1) + 0.5 * rho * (u * u + v * v))
    speed = 0.0
    for base, ox, oy in ((4, 0.0, 0.0), (8, 0.0, 0.5), (12, 0.5, 0.0)):
        for k, f in enumerate(fn(x + ox * g.h, y + oy * g.h)):
            s[base + k] = f
        rho, u, v, p = s[base:base + 4]
        speed = max(speed, float((torch.sqrt(u * u + v * v) + torch.sqrt(GAMMA * p / rho)).max()))
    return g, s, CFL * g.h / speed


def _cotangent(case, seed):
    """A seeded adjoint of the state, as a loss over a whole field gives it."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed + 1)
    return torch.randn((16, case["ny"], case["nx"]), dtype=torch.float64, device="cuda",
                       generator=g)


def _members(case):
    """An ensemble's members, one case each: uneven sizes from the smallest grid up
    to `most`, doubling, in an order that depends on the number of members alone."""
    r, n, sizes = _rng(case["members"]), case["nx"], []
    while n <= case["most"]:
        sizes.append(n)
        n *= 2
    return [dict(case, nx=s, ny=s) for s in (int(r.choice(sizes)) for _ in range(case["members"]))]


def _problems(case, seed):
    probs, dts = [], []
    for m, c in enumerate(_members(case)):
        g, s, dt = _state(c, seed, m)
        probs.append(_Problem(g, GAMMA, s.cpu().numpy()))
        dts.append(dt)
    return probs, dts


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        probs, dts = _problems(case, seed)
        return dict(case=case, problems=probs, dts=dts)
    g, s, dt = _state(case, seed)
    st = dict(case=case, grid=g, dt=dt, x0=s)
    if kind == "gradient":
        st["g"] = _cotangent(case, seed)
        return st
    st["solver"] = af.Solver(g, GAMMA, s, precision=case["precision"], variant=case["variant"],
                             stream=torch.cuda.current_stream())
    if kind == "host":
        st["x0"] = s.cpu().pin_memory()
        st["out"] = torch.empty_like(st["x0"], pin_memory=True)
    elif kind == "step":
        st["out"] = torch.empty_like(s)
    elif kind == "adjoint":
        st["g"] = _cotangent(case, seed)
        st["out"] = torch.empty_like(s)
    return st


def _of_mode(case, x):
    return x if case["precision"] == "fp64" else x.to(torch.float32)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("step", "host"):
        s = state["solver"]
        s.set_state(state["x0"])
        s.step(state["dt"], case["steps"])
        return _of_mode(case, s.state(state["out"]))
    if kind == "adjoint":
        lam = state["solver"].adjoint(state["dt"], state["g"], state["out"])
        return _of_mode(case, lam)
    if kind == "gradient":
        x0 = state["x0"].detach().requires_grad_(True)
        xn = rollout(x0, state["grid"], GAMMA, state["dt"], case["steps"],
                     checkpoint_every=case["every"], precision=case["precision"],
                     variant=case["variant"])
        xn.backward(state["g"])
        return {"state": _of_mode(case, xn.detach()), "grad": _of_mode(case, x0.grad)}
    if kind == "invariants":
        return state["solver"].invariants()
    b = af.Batch(state["problems"], precision=case["precision"], variant=case["variant"])
    b.step(state["dts"], case["steps"])
    out = [torch.from_numpy(b.state(k)).to(torch.float32) for k in range(case["members"])]
    b.close()
    return out


# Operations of one step per cell and bytes of one state, both of one cell
# (the sixteen float64 planes of the API).
_OPS = {"tai": 2233, "rb": 2000, "fc": 20000}


def work(case):
    kind, prec = case["kind"], case["precision"]
    cells = case["nx"] * case["ny"]
    if kind == "ensemble":
        cells = sum(c["nx"] * c["ny"] for c in _members(case))
    state = 128.0 * cells
    back = state if prec == "fp64" else state / 2
    ops = _OPS[case["variant"]] * cells
    if kind in ("step", "host", "ensemble"):
        # the averages' and points' planes go through HBM once each way per step
        # where a state is larger than the L2 cache can hold
        plane = 8 if prec == "fp64" else 4
        step = 2 * (20 if prec == "fp32_comp" else 16) * plane * cells
        return {"bytes": state + back + (case["steps"] * step if step > 1.3e8 else 0),
                "flops": ops * case["steps"]}
    if kind == "adjoint":
        return {"bytes": 2 * state + back, "flops": 3.0 * ops}
    if kind == "gradient":
        return {"bytes": 2 * state + 2 * back, "flops": 5.0 * ops * case["steps"]}
    return {"bytes": (160.0 if prec == "fp32_comp" else 64.0 if prec == "fp32" else 128.0) * cells,
            "flops": 250.0 * cells}


# ---- the scheme in float64 torch ----------------------------------------------------
# All nodes of the Q2 reconstruction on the lattice of half cells, shape
# (4, 2 ny, 2 nx): (rho, u, v, p) at vertices (even, even), x-edge midpoints
# (odd row, even column), y-edge midpoints (even row, odd column) and centres.
_FAMILIES = ((0, 0), (0, 1), (1, 0), (1, 1))  # column and row parity: V, E_v, E_h, C


def _prim(u):
    r = u[0]
    a, b = u[1] / r, u[2] / r
    return torch.stack([r, a, b, (GAMMA - 1) * (u[3] - 0.5 * (u[1] * a + u[2] * b))])


def _cons(w):
    r, u, v, p = w
    return torch.stack([r, r * u, r * v, p / (GAMMA - 1) + 0.5 * r * (u * u + v * v)])


def _next(x, axis):
    return torch.roll(x, -1, dims=axis)


def _lattice(st):
    avg, vt, ev, eh = st[0:4], st[4:8], st[8:12], st[12:16]
    cv = _cons(vt)
    corners = cv + _next(cv, 2) + _next(cv, 1) + _next(_next(cv, 2), 1)
    ce, ch = _cons(ev), _cons(eh)
    edges = ce + _next(ce, 2) + ch + _next(ch, 1)
    centre = _prim(2.25 * avg - corners / 16 - edges / 4)
    rows = [torch.stack([vt, eh], 3).flatten(2), torch.stack([ev, centre], 3).flatten(2)]
    return torch.stack(rows, 2).flatten(1, 2)


def _zeta(j):
    return math.sqrt(math.pi) * math.gamma((j + 1) / 2) / math.gamma(j / 2 + 1)


def _block(a, b, t0, t1):
    """The frozen acoustic operator on the wedge t0 < theta < t1 and the monomial
    X^a Y^b, weight r^(a+b), as a (pi, u, v) x (pi, u, v) matrix."""
    x, w = np.polynomial.legendre.leggauss(40)
    t = 0.5 * (t1 - t0) * x + 0.5 * (t1 + t0)

    def mu(m, n):
        return float(np.sum(0.5 * (t1 - t0) * w * np.cos(t) ** m * np.sin(t) ** n))

    q = a + b
    chi = 1.0 if q == 0 else 1 + 1.0 / q
    e = q + 1 + 3 * chi
    m = mu(a, b) * _zeta(q + 1)
    px, py = ((q + 2) * mu(a + i, b + j) * _zeta(q + 2) for i, j in ((1, 0), (0, 1)))
    xx, xy, yy = (mu(a + i, b + j) * _zeta(q + 3) for i, j in ((2, 0), (1, 1), (0, 2)))
    k = np.array([[(q + 1) * m, -px, -py], [-px, e * xx - chi * m, e * xy],
                  [-py, e * xy, e * yy - chi * m]]) / (4 * math.pi)
    if q == 0:
        k += (2.0 / 3.0) * (t1 - t0) / (2 * math.pi) * np.diag([0.0, 1.0, 1.0])
    return k


_STENCILS = {}


def _stencils(col, row):
    """Weights (4 powers of r, 3 outputs, 3 inputs, 5, 5) of a node family."""
    if (col, row) in _STENCILS:
        return _STENCILS[col, row]
    h = math.pi / 2
    wedges = {(0, 0): [(0, h, 0, 0), (h, 2 * h, 1, 0), (2 * h, 3 * h, 1, 1), (3 * h, 4 * h, 0, 1)],
              (0, 1): [(-h, h, 0, .5), (h, 3 * h, 1, .5)], (1, 0): [(0, 2 * h, .5, 0),
              (2 * h, 4 * h, .5, 1)], (1, 1): [(0, 4 * h, .5, .5)]}[col, row]
    out = np.zeros((5, 3, 3, 5, 5))
    for t0, t1, ox, oy in wedges:
        xs, ys = (np.array([0, .5, 1]) - o for o in (ox, oy))
        # monomial coefficients [power, node] of the Lagrange basis on these nodes
        lx, ly = np.linalg.inv(np.vander(xs, 3, True)), np.linalg.inv(np.vander(ys, 3, True))
        for a in range(3):
            for b in range(3):
                k = _block(a, b, t0, t1)
                for i in range(3):
                    for j in range(3):
                        out[a + b, :, :, int(round(2 * ys[j])) + 2, int(round(2 * xs[i])) + 2] += \
                            lx[a, i] * ly[b, j] * k
    _STENCILS[col, row] = out[1:]  # the power 0 is the identity
    return _STENCILS[col, row]


def _increments(lat, dth):
    """Acoustic increments (du, dv, dp) of all lattice nodes, for dt / 2 and dt."""
    ny2, nx2 = lat.shape[1:]
    src = torch.stack([lat[3], lat[1], lat[2]])[None]
    pad = F.pad(src, (2, 2, 2, 2), mode="circular")
    out = [torch.zeros((3, ny2 // 2, 2, nx2 // 2, 2), dtype=lat.dtype, device=lat.device)
           for _ in range(2)]
    parts = [[None] * 4, [None] * 4]
    for f, (col, row) in enumerate(_FAMILIES):
        w = torch.as_tensor(_stencils(col, row), dtype=lat.dtype, device=lat.device)
        own = lat[:, row::2, col::2]
        rho, p = own[0], own[3]
        c = torch.sqrt(GAMMA * p / rho)
        z = rho * c
        # the node's own value is subtracted: the weights of each power sum to 0
        x = pad[:, :, row:row + ny2 + 3, col:col + nx2 + 3]
        wp, wu = w.clone(), w.clone()
        wp[:, :, 1:], wu[:, :, 0] = 0, 0
        gp = F.conv2d(x, wp.reshape(12, 3, 5, 5), stride=2)[0].reshape(4, 3, *p.shape)
        gu = F.conv2d(x, wu.reshape(12, 3, 5, 5), stride=2)[0].reshape(4, 3, *p.shape)
        for s in range(2):
            r = c * dth * (0.5 if s == 0 else 1.0)
            d = [0, 0, 0]
            for q in (3, 2, 1, 0):
                d[0] = r * (d[0] + gp[q, 1] / z + gu[q, 1])
                d[1] = r * (d[1] + gp[q, 2] / z + gu[q, 2])
                d[2] = r * (d[2] + gp[q, 0] + z * gu[q, 0])
            parts[s][f] = torch.stack(d)
    for s in range(2):
        v, ev, eh, c = parts[s]
        rows = [torch.stack([v, eh], 3).flatten(2), torch.stack([ev, c], 3).flatten(2)]
        out[s] = torch.stack(rows, 2).flatten(1, 2)
    return out


def _q2(lat, col, row, dx, dy):
    """Q2 reconstruction of the lattice fields at the family's points moved by
    (dx, dy) cells, and a function that evaluates further fields there."""
    ny2, nx2 = lat.shape[1:]
    fx, fy = 0.5 * col + dx, 0.5 * row + dy
    cx, cy = torch.floor(fx.detach()), torch.floor(fy.detach())
    s, t = 2 * (fx - cx) - 1, 2 * (fy - cy) - 1
    lx = (0.5 * s * (s - 1), 1 - s * s, 0.5 * s * (s + 1))
    ly = (0.5 * t * (t - 1), 1 - t * t, 0.5 * t * (t + 1))
    i = torch.arange(nx2 // 2, device=lat.device)[None, :] + cx.long()
    j = torch.arange(ny2 // 2, device=lat.device)[:, None] + cy.long()

    def at(f):
        out = 0
        for b in range(3):
            for a in range(3):
                idx = ((2 * j + b) % ny2) * nx2 + (2 * i + a) % nx2
                out = out + lx[a] * ly[b] * f.flatten(1)[:, idx]
        return out

    return at(lat), at


def _flux(w, axis):
    r, u, v, p = w
    n = u if axis == 0 else v
    m = r * n
    e = p * GAMMA / (GAMMA - 1) + 0.5 * r * (u * u + v * v)
    return torch.stack([m, m * u + (p if axis == 0 else 0), m * v + (p if axis == 1 else 0), n * e])


def _step(st, h, dt, variant):
    lat = _lattice(st)
    inc = _increments(lat, dt / h)
    levels = [[st[4:8], st[8:12], st[12:16]]]
    for s in range(2):
        th = dt / h * (0.5 if s == 0 else 1.0)
        new = []
        for f, (col, row) in enumerate(_FAMILIES[:3]):
            w = st[4 + 4 * f:8 + 4 * f]
            w1, _ = _q2(lat, col, row, -th * w[1], -th * w[2])
            wf, at = _q2(lat, col, row, -th * w1[1], -th * w1[2])
            if variant == "tai":
                d, rc, pc = at(inc[s]), wf[0], wf[3]
            else:
                d, rc, pc = inc[s][:, row::2, col::2], w[0], w[3]
            new.append(torch.stack([wf[0] + d[2] * rc / (GAMMA * pc), wf[1] + d[0], wf[2] + d[1],
                                    wf[3] + d[2]]))
        levels.append(new)
    fx = gy = 0
    for wt, (v, ev, eh) in zip((1, 4, 1), levels):
        a, b = _flux(v, 0), _flux(v, 1)
        fx = fx + wt * (a + 4 * _flux(ev, 0) + _next(a, 1))
        gy = gy + wt * (b + 4 * _flux(eh, 1) + _next(b, 2))
    lam = dt / (36 * h)
    avg = st[0:4] - lam * (_next(fx, 2) - fx) - lam * (_next(gy, 1) - gy)
    return torch.cat([avg] + levels[2])


def _entropy(r, p):
    return -r * torch.log(p / r ** GAMMA)


def _invariants(st, h):
    lat = _lattice(st)
    a, b = st[0:4], _prim(st[0:4])
    w = torch.tensor([1.0, 2.0], dtype=st.dtype, device=st.device)
    wx, wy = w.repeat(st.shape[2]), w.repeat(st.shape[1])
    area = h * h
    simpson = (_entropy(lat[0], lat[3]) * wy[:, None] * wx[None, :]).sum() / 9
    v, e, eh = st[4:8], st[8:12], st[12:16]
    left, low = v[2] + 4 * e[2] + _next(v[2], 0), v[1] + 4 * eh[1] + _next(v[1], 1)
    curl = h / 6 * ((_next(left, 1) - left) - (_next(low, 0) - low)).sum()
    speed = torch.sqrt(lat[1] ** 2 + lat[2] ** 2) + torch.sqrt(GAMMA * lat[3] / lat[0])
    vals = [area * a[k].sum() for k in range(4)]
    vals += [area * simpson, area * _entropy(b[0], b[3]).sum(),
             area * (0.5 * (a[1] ** 2 + a[2] ** 2) / a[0]).sum(), speed.max(), lat[0].min(),
             lat[3].min(), curl]
    return np.array([float(x) for x in vals] + [0.0])


def exact(case, seed):
    kind = case["kind"]
    if case["variant"] == "fc":
        return None  # its disk integrals take minutes in plain torch
    if kind == "ensemble":
        if case["members"] * case["steps"] > 450:
            return None
        outs = []
        with torch.no_grad():
            for m, c in enumerate(_members(case)):
                g, s, dt = _state(c, seed, m)
                for _ in range(case["steps"]):
                    s = _step(s, g.h, dt, case["variant"])
                outs.append(s.cpu())
        return outs
    g, s, dt = _state(case, seed)
    if kind == "invariants":
        return _invariants(s, g.h)
    states = [s]
    with torch.no_grad():
        for _ in range(case["steps"]):
            s = _step(s, g.h, dt, case["variant"])
            if kind == "gradient":
                states.append(s)
    if kind == "host":
        return s.cpu()
    if kind == "step":
        return s
    lam = _cotangent(case, seed)
    begin = states[:-1] if kind == "gradient" else [states[0]]
    for x in reversed(begin):
        x = x.detach().requires_grad_(True)
        lam, = torch.autograd.grad(_step(x, g.h, dt, case["variant"]), x, lam)
    return lam if kind == "adjoint" else {"state": states[-1], "grad": lam}
