"""Timed cases of the solver: what a user has it do, through the library's public entry points.

A case is one solve (or one batch of solves) advanced by a few steps: the initial planes are on the
GPU, the solver object exists (a user's program keeps it from call to call), and one pass loads the
state, steps it and copies the new state into a device tensor.  The sizes are those of the package's
workloads and of the paper's tests (Sec. 4): 1D tubes and waves of about a hundred cells, small
and ragged 2D grids, the 200^2 pulses, 512^2 and 2048^2 vortices, the 1024x512 shock-vortex, and
batches of many uneven grids.  Both reconstruction orders, both variable sets, inviscid and viscous
flow and all four boundary types occur.

``exact`` is the scheme written out plainly in 64-bit torch arithmetic.
"""
import math

import numpy as np
import torch

from paper_2001_01570_gb300 import cgks

PERIODIC, REFLECT, INFLOW, OUTFLOW = 0, 1, 2, 3
GAMMA = 1.4
DEVICE = torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")


def listed():
    return [
        # the paper's 1D accuracy test: one small latency-bound solve
        dict(name="wave1d_100", kind="wave1d", nx=100, steps=60),
        # a shock tube in characteristic variables, odd size
        dict(name="sod1d_401_char", kind="sod", nx=401, steps=40, char=True),
        # the smallest grid of the batched and served streams, run alone
        dict(name="pulse_64", kind="pulse", nx=64, ny=64, steps=20),
        # ragged small viscous flow with the 6th-order reconstruction
        dict(name="viscous_97x61_o6", kind="viscous", nx=97, ny=61, steps=10, order=6),
        # the caller's own device buffer, no allocation inside the call
        dict(name="noalloc_vortex_128", kind="vortex", nx=128, ny=128, steps=8, entry="noalloc"),
        # Mach-2.9 regular reflection in characteristic variables (paper Sec. 4: 200 x 50)
        dict(name="reflection_200x50_char", kind="reflection", nx=200, ny=50, steps=16, char=True),
        # acoustic, entropy and vorticity pulses (paper Sec. 4.6)
        dict(name="pulses_200", kind="pulse", nx=200, ny=200, steps=10),
        dict(name="vortex_512", kind="vortex", nx=512, ny=512, steps=4),
        dict(name="shock_vortex_1024x512", kind="shock_vortex", nx=1024, ny=512, steps=2),
        # the largest single grid of the benchmark
        dict(name="vortex_2048", kind="vortex", nx=2048, ny=2048, steps=2),
        # many uneven 2D grids in one persistent launch per kernel and stage
        dict(name="batch_40_pulses", kind="batch", count=40, nmin=64, nmax=512, steps=4),
        # many tiny 1D solves (the coarse meshes of the paper's 1D acoustic wave)
        dict(name="batch1d_256_waves", kind="batch1d", count=256, nmin=12, nmax=48, steps=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["wave1d", "sod", "pulse", "pulse", "vortex", "vortex", "viscous", "noalloc", "reflection",
                       "shock_vortex", "batch", "batch1d"])
    char, order = rng.random() < 0.25, 6 if rng.random() < 0.25 else 8
    if kind in ("wave1d", "sod"):
        return dict(kind=kind, nx=_log(rng, 24, 1000), steps=rng.randint(20, 60), char=char, order=order)
    if kind == "noalloc":
        return dict(kind=rng.choice(["vortex", "pulse"]), nx=_log(rng, 48, 250), ny=_log(rng, 48, 250),
                    steps=rng.randint(4, 10), entry="noalloc", order=order)
    if kind in ("batch", "batch1d"):
        lo, hi = (64, 512) if kind == "batch" else (12, 48)
        return dict(kind=kind, count=_log(rng, 8, 40) if kind == "batch" else _log(rng, 64, 256), nmin=lo, nmax=hi,
                    steps=rng.randint(2, 4) if kind == "batch" else rng.randint(5, 10), order=order)
    if kind == "reflection":
        nx = _log(rng, 60, 800)
        return dict(kind=kind, nx=nx, ny=max(12, nx // 4 + rng.randint(-2, 2)), steps=rng.randint(4, 16), char=char)
    if kind == "shock_vortex":
        nx = _log(rng, 96, 1024)
        return dict(kind=kind, nx=nx, ny=max(24, nx // 2 + rng.randint(-3, 3)), steps=2, char=char, order=order)
    nx = _log(rng, 48, 2048 if kind == "vortex" else 700)
    ny = max(32, min(2048, int(nx * rng.uniform(0.5, 1.0))))
    steps = 2 if nx * ny > 300000 else rng.randint(4, 12)
    return dict(kind=kind, nx=nx, ny=ny, steps=steps, char=char and nx < 700, order=order)


# ----------------------------------------------------------------------------- initial states
_GX, _GW = (a * 0.5 for a in np.polynomial.legendre.leggauss(6))


def _cons(q):
    rho, u, v, p = q
    return torch.stack([rho, rho * u, rho * v, p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)])


def _planes(fun, box, nx, ny):
    """Cell averages (6 x 6 Gauss points) and cell-averaged gradients (divergence theorem) of fun."""
    x0, x1, y0, y1 = box
    dx, dy = (x1 - x0) / nx, (y1 - y0) / ny
    x = (x0 + (torch.arange(nx, dtype=torch.float64, device=DEVICE) + 0.5) * dx)[None, :].expand(ny, nx)
    y = (y0 + (torch.arange(ny, dtype=torch.float64, device=DEVICE) + 0.5) * dy)[:, None].expand(ny, nx)
    W = torch.zeros(12, ny, nx, dtype=torch.float64, device=DEVICE)
    half = 0.5 - 1e-9
    for a, wa in zip(_GX, _GW):
        for b, wb in zip(_GX, _GW) if ny > 1 else [(0.0, 1.0)]:
            W[:4] += wa * wb * _cons(fun(x + a * dx, y + b * dy))
        if ny == 1:
            continue
        W[4:8] += wa / dx * (_cons(fun(x + half * dx, y + a * dy)) - _cons(fun(x - half * dx, y + a * dy)))
        W[8:] += wa / dy * (_cons(fun(x + a * dx, y + half * dy)) - _cons(fun(x + a * dx, y - half * dy)))
    if ny == 1:
        W[4:8] = (_cons(fun(x + half * dx, y)) - _cons(fun(x - half * dx, y))) / dx
    return W


def _flow(case, rng):
    """(domain, boundary types, inflow states per side, other options, fun(x, y) -> rho, u, v, p)."""
    kind, nx, ny = case["kind"], case["nx"], case.get("ny", 1)
    one = (1.0, 0.0, 0.0, 1.0)
    if kind == "wave1d":
        amp, ph = rng.uniform(0.1, 0.25), rng.uniform(0.0, 2.0)
        return (0.0, 2.0, 0.0, 1.0), (0, 0, 0, 0), (one,) * 4, dict(cfl=0.3), lambda x, y: (
            1.0 + amp * torch.sin(math.pi * (x - ph)), torch.ones_like(x), torch.zeros_like(x), torch.ones_like(x))
    if kind == "sod":
        rl, pl = rng.uniform(0.8, 1.2), rng.uniform(0.8, 1.2)
        cut = (nx // 2) / nx
        return (0.0, 1.0, 0.0, 1.0), (OUTFLOW, OUTFLOW, 0, 0), (one,) * 4, {}, lambda x, y: (
            torch.where(x < cut, rl, 0.125).to(x), torch.zeros_like(x), torch.zeros_like(x),
            torch.where(x < cut, pl, 0.1).to(x))
    if kind == "pulse":
        # weak acoustic pulse (dx = 1) on a gas at rest, as in the batched and served streams
        amp, b = 10.0 ** rng.uniform(-5.0, -3.0), rng.uniform(3.0, 10.0)
        cx, cy = rng.uniform(0, nx), rng.uniform(0, ny)

        def fun(x, y):
            rx = torch.remainder(x - cx + 0.5 * nx, nx) - 0.5 * nx
            ry = torch.remainder(y - cy + 0.5 * ny, ny) - 0.5 * ny
            o = torch.ones_like(x)
            return o, 0 * o, 0 * o, 1.0 / GAMMA + amp * torch.exp(-math.log(2.0) * (rx * rx + ry * ry) / (b * b))
        return (0.0, float(nx), 0.0, float(ny)), (0, 0, 0, 0), (one,) * 4, {}, fun
    if kind in ("vortex", "viscous"):
        Lx, Ly, s = 10.0, 10.0 * ny / nx, rng.uniform(3.0, 5.0)
        cx, cy = rng.uniform(0, Lx), rng.uniform(0, Ly)

        def fun(x, y):
            rx = torch.remainder(x - cx + 0.5 * Lx, Lx) - 0.5 * Lx
            ry = torch.remainder(y - cy + 0.5 * Ly, Ly) - 0.5 * Ly
            e = torch.exp(0.5 * (1.0 - rx * rx - ry * ry))
            T = 1.0 - (GAMMA - 1.0) * s * s / (8.0 * GAMMA * math.pi ** 2) * e * e
            rho = T ** (1.0 / (GAMMA - 1.0))
            return rho, 1.0 - s / (2 * math.pi) * e * ry, 1.0 + s / (2 * math.pi) * e * rx, rho * T
        return (0.0, Lx, 0.0, Ly), (0, 0, 0, 0), (one,) * 4, dict(mu=0.002) if kind == "viscous" else {}, fun
    if kind == "shock_vortex":
        m, vm, a, b = rng.uniform(1.05, 1.5), 0.3, 0.05, 0.2
        c1 = math.sqrt(GAMMA)
        cut = round(nx / 4) * 2.0 / nx                       # the shock stands on a face
        r2 = (GAMMA + 1) * m * m / ((GAMMA - 1) * m * m + 2)
        p2, u1 = 1 + 2 * GAMMA / (GAMMA + 1) * (m * m - 1), m * c1
        cx, cy, k = 0.5 * cut, rng.uniform(0.4, 0.6), vm * c1 * a / (a * a - b * b)

        def fun(x, y):
            rx, ry = x - cx, y - cy
            r = torch.sqrt(rx * rx + ry * ry).clamp_min(1e-12)

            def temp(q):
                return 1 - (GAMMA - 1) / GAMMA * k * k * (b ** 4 / (2 * q * q) - q * q / 2 - 2 * b * b * torch.log(b / q))
            core = temp(torch.full_like(r, a)) - (GAMMA - 1) / GAMMA * (vm * c1) ** 2 * (a * a - r * r) / (2 * a * a)
            T = torch.where(r <= a, core, torch.where(r <= b, temp(r), torch.ones_like(r)))
            vt = torch.where(r <= a, vm * c1 * r / a, torch.where(r <= b, k * (r - b * b / r), torch.zeros_like(r)))
            up, rho = x < cut, T ** (1.0 / (GAMMA - 1.0))
            return (torch.where(up, rho, r2), torch.where(up, u1 - vt * ry / r, u1 / r2),
                    torch.where(up, vt * rx / r, 0.0), torch.where(up, rho * T, p2))
        return ((0.0, 2.0, 0.0, 1.0), (INFLOW, OUTFLOW, REFLECT, REFLECT), ((1.0, u1, 0.0, 1.0),) * 4, {}, fun)
    # regular reflection of an oblique shock: free stream at the left, the state behind it through the top
    m, ang = rng.uniform(2.6, 2.9), math.radians(29.0)
    un, ut = m * math.sin(ang), m * math.cos(ang)
    r2 = (GAMMA + 1) * un * un / ((GAMMA - 1) * un * un + 2)
    p2, un2 = (1 + 2 * GAMMA / (GAMMA + 1) * (un * un - 1)) / GAMMA, un / r2
    free = (1.0, m, 0.0, 1.0 / GAMMA)
    post = (r2, ut * math.cos(ang) + un2 * math.sin(ang), un2 * math.cos(ang) - ut * math.sin(ang), p2)
    # the incident shock is there (steps on cell faces), the reflected one still has to form
    sl = math.tan(ang)

    def fun(x, y):
        above = (torch.floor(y * ny) + 0.5) / ny > 1.0 - sl * ((torch.floor(x * nx / 4.0) + 0.5) * 4.0 / nx)
        return tuple(torch.where(above, b, a).to(x) for a, b in zip(free, post))
    return (0.0, 4.0, 0.0, 1.0), (INFLOW, OUTFLOW, REFLECT, INFLOW), (free, free, free, post), {}, fun


def _members(case, seed):
    """The single-grid cases of a batch; the sizes depend on the case alone, the flows on the seed."""
    if case["kind"] not in ("batch", "batch1d"):
        return [case]
    rng, out = np.random.default_rng(1570), []
    for _ in range(case["count"]):
        n = int(round(math.exp(rng.uniform(math.log(case["nmin"]), math.log(case["nmax"])))))
        out.append(dict(case, kind="pulse", nx=n, ny=n) if case["kind"] == "batch" else dict(case, kind="wave1d", nx=n))
    return out


def _is_1d(case):
    return case["kind"] in ("wave1d", "sod")


def _setup(case, rng):
    """(arguments of cgks.make_problem, 2D planes (12, ny, nx)) of one grid."""
    box, bc, inflow, more, fun = _flow(case, rng)
    nx, ny = case["nx"], case.get("ny", 1)
    kw = dict(dim=1 if _is_1d(case) else 2, nx=nx, ny=ny, x0=box[0], x1=box[1], y0=box[2], y1=box[3], gamma=GAMMA,
              cfl=0.5, bc=bc, inflow=inflow, recon_vars=1 if case.get("char") else 0, order=case.get("order", 8))
    kw.update(more)
    return kw, _planes(fun, box, nx, ny)


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    grids = []
    for c in _members(case, seed):
        kw, W = _setup(c, rng)
        if kw["dim"] == 1:
            W = W[[0, 1, 3, 4, 5, 7], 0].contiguous()
        prob = cgks.make_problem(**kw)
        noalloc = case.get("entry") == "noalloc"
        grids.append((prob if noalloc else cgks.Solver(prob), W, torch.empty_like(W)))
    return dict(case=dict(case), grids=grids)


def run(state):
    case, grids = state["case"], state["grids"]
    if case.get("entry") == "noalloc":
        prob, W, out = grids[0]
        out.copy_(W)
        return [out, cgks.cgks_step_noalloc(prob, out, case["steps"])]
    for s, W, _ in grids:
        cgks.cgks_set_state(s.handle, W)
    if case["kind"] in ("batch", "batch1d"):
        cgks.cgks_batch_step([s.handle for s, _, _ in grids], case["steps"])
    else:
        cgks.cgks_step(grids[0][0].handle, case["steps"])
    times = [cgks.cgks_get_state(s.handle, out)[0] for s, _, out in grids]
    if len(grids) > 1:
        return [torch.cat([out.flatten() for _, _, out in grids]), np.array(times)]
    return [grids[0][2], times[0]]


def work(case):
    cells = [c["nx"] * c.get("ny", 1) for c in _members(case, 0)]
    planes = 6 if case["kind"] in ("wave1d", "sod", "batch1d") else 12
    # per cell and step: the operations of the scheme's formulas (both stages; 1D: one face row and
    # one face per cell instead of two)
    flops = 18068.0 if planes == 12 else 9034.0
    return {"bytes": 2.0 * 8 * planes * sum(cells), "flops": flops * sum(cells) * case["steps"]}


# ----------------------------------------------------------------------------- the scheme in 64 bits
def _fit(cells, slopes):
    """Matrix from the stencil data (Q_{i-1..i+2} - Q_i, h Q'_{i-1..i+2}) to the monomial coefficients
    (xi = (x - x_i)/h) of the polynomial with these cell averages and cell-averaged slopes."""
    rows = [(0, c) for c in cells] + [(1, c) for c in slopes]
    n = len(rows)
    A, pick = np.zeros((n, n)), np.zeros((n, 8))
    for r, (kind, c) in enumerate(rows):
        lo, hi = c - 0.5, c + 0.5
        for m in range(n):
            A[r, m] = (hi ** (m + 1) - lo ** (m + 1)) / (m + 1) if kind == 0 else hi ** m - lo ** m
        pick[r, 4 * kind + c + 1] = 1.0
    return np.linalg.solve(A, pick)


def _roughness(n):
    """Matrix of sum_r int_{-1/2}^{1/2} (d^r q / dxi^r)^2 on monomial coefficients."""
    H, D = np.zeros((n, n)), np.eye(n)
    G = np.array([[(0.5 ** (i + j + 1) - (-0.5) ** (i + j + 1)) / (i + j + 1) for j in range(n)] for i in range(n)])
    step = np.diag(np.arange(1.0, n), 1)
    for _ in range(1, n):
        D = step @ D
        H += D.T @ G @ D
    return H


_STENCILS = [((-1, 0), (-1,)), ((-1, 0, 1), ()), ((0, 1, 2), (2,)), ((-1, 0, 1), ()), ((0, 1, 2), ()),
             ((-1, 0, 1), (-1, 0)), ((0, 1, 2), (1, 2))]
_FITS = [_fit(*s) for s in _STENCILS]
_BETA_FITS = [_FITS[0], _fit((-1, 0, 1), (-1,))] + _FITS[2:]
_WEIGHTS = {8: np.array([3, 5, 8, 7, 7, 34, 34]) / 98.0, 6: np.array([3, 5, 8, 7, 7, 20, 20]) / 70.0}


def _apply(row, data):
    acc = None
    for c, d in zip(row, data):
        if abs(c) > 1e-13:
            acc = c * d if acc is None else acc + c * d
    return torch.zeros_like(data[0]) if acc is None else acc


def _weno(Q, S, order, eps):
    """Left value and h * slope at x_{i+1/2} from Q, S = values and h * slopes of cells i-1..i+2."""
    data = [Q[0] - Q[1], torch.zeros_like(Q[1]), Q[2] - Q[1], Q[3] - Q[1]] + list(S)
    beta, val, slope = [], [], []
    for M, B in zip(_FITS, _BETA_FITS):
        n = M.shape[0]
        val.append(_apply(0.5 ** np.arange(n) @ M, data))
        slope.append(_apply((np.arange(n) * 0.5 ** np.maximum(np.arange(n) - 1, 0)) @ M, data))
        H = _roughness(B.shape[0])
        w, V = np.linalg.eigh(H)
        forms = [(lam, _apply(V[:, k] @ B, data)) for k, lam in enumerate(w) if lam > 1e-12]
        beta.append(sum(lam * f * f for lam, f in forms))
    Z = (3.0 * (beta[0] - beta[4]) + (beta[4] - beta[3])).abs()
    alpha = [d * (1.0 + Z / (b + eps)) for d, b in zip(_WEIGHTS[order], beta)]
    total = sum(alpha)
    return Q[1] + sum(a * v for a, v in zip(alpha, val)) / total, sum(a * s for a, s in zip(alpha, slope)) / total


def _weno_pair(Q, S, order, eps):
    vl, sl = _weno(Q, S, order, eps)
    vr, sr = _weno(Q[::-1], [-s for s in S[::-1]], order, eps)
    return vl, sl, vr, -sr


def _linear(Q, S, order):
    a, b, c, d = Q
    A, B, C, D = S
    if order == 6:
        return (((a + d) + 29 * (b + c)) / 60 + (B - C) / 5, 2.25 * (c - b) + (d - a) / 36 - 2 * (B + C) / 3,
                ((b + c) - (a + d)) / 4 - 1.5 * (B - C))
    return ((25 * (a + d) + 185 * (b + c) + 6 * (A - D) + 102 * (B - C)) / 420,
            (270 * (c - b) + 14 * (d - a) - 3 * (A + D) - 99 * (B + C)) / 108,
            (b + c) - (a + d) - (A - D) / 4 - 2.25 * (B - C))


def _char_pair(Q, S, order, eps):
    """The pair in characteristic variables at the mean of the two cells sharing the face."""
    W = 0.5 * (Q[1] + Q[2])
    rho, U, V = W[0], W[1] / W[0], W[2] / W[0]
    q2 = U * U + V * V
    p = (GAMMA - 1) * (W[3] - 0.5 * rho * q2)
    c, H = torch.sqrt(GAMMA * p / rho), (W[3] + p) / rho
    b2 = (GAMMA - 1) / (c * c)
    b1, z, o = 0.5 * b2 * q2, torch.zeros_like(U), torch.ones_like(U)
    L = [[0.5 * (b1 + U / c), -0.5 * (b2 * U + 1 / c), -0.5 * b2 * V, 0.5 * b2], [1 - b1, b2 * U, b2 * V, -b2],
         [-V, z, o, z], [0.5 * (b1 - U / c), -0.5 * (b2 * U - 1 / c), -0.5 * b2 * V, 0.5 * b2]]
    R = [[o, o, z, o], [U - c, U, z, U + c], [V, V, o, V], [H - U * c, 0.5 * q2, V, H + U * c]]
    mul = lambda M, w: torch.stack([sum(M[r][k] * w[k] for k in range(4)) for r in range(4)])  # noqa: E731
    got = _weno_pair([mul(L, q) for q in Q], [mul(L, s) for s in S], order, eps)
    return tuple(mul(R, g) for g in got)


def _weno5(v):
    """Slopes at the centre and second differences of the three quadratics on five segment means."""
    D = [3 * v[2] - 4 * v[1] + v[0], v[3] - v[1], 4 * v[3] - v[4] - 3 * v[2]]
    s = [v[0] - 2 * v[1] + v[2], v[1] - 2 * v[2] + v[3], v[2] - 2 * v[3] + v[4]]
    return D, s


def _along(rec, T, kw, h):
    """Gauss-point data along the faces from the rows' line averages; rec maps a name to (4, T + 4, F)."""
    eps = kw["weno_eps"]
    at = lambda f, o: rec[f][:, 2 + o: 2 + o + T]  # noqa: E731
    v = [at("V", o) for o in range(-2, 3)]
    n = [at("N", o) for o in range(-2, 3)]
    D, s = _weno5(v)
    e = [13.0 / 12.0 * b * b + 0.25 * a * a + eps for a, b in zip(D, s)]
    Z = (e[0] - e[2]).abs()
    dl, dh = 7.0 / 36.0 - math.sqrt(3.0) / 1080.0, 7.0 / 36.0 + math.sqrt(3.0) / 1080.0

    def three(f):
        m, z, p = (at(f, o) for o in (-1, 0, 1))
        a, b = z - m, p - z
        ea, eb = a * a + eps, b * b + eps
        zz = (ea - eb).abs()
        wa, wb = 0.5 * (1 + zz / ea), 0.5 * (1 + zz / eb)
        return z, (wa * a + wb * b) / (wa + wb)
    Lv, Ls = three("L")
    Rv, Rs = three("R")

    def quartic(m, eta):
        S1, S2, A1, A2 = m[3] + m[1], m[4] + m[0], m[3] - m[1], m[4] - m[0]
        val = m[2] - (S2 - 4 * S1 + 6 * m[2]) / 4320 + eta * (50 * A1 - 7 * A2) / 72
        d1 = (8 * A1 - A2) / 12 + eta * (13 * S1 - S2 - 24 * m[2]) / 9
        d2 = (16 * S1 - S2 - 30 * m[2]) / 12 + eta * (A2 - 2 * A1) / 2
        return val, d1 / h, d2 / (h * h)

    for sign in (-1.0, 1.0):
        eta = sign / (2.0 * math.sqrt(3.0))
        w = (dl, 11.0 / 18.0, dh) if sign > 0 else (dh, 11.0 / 18.0, dl)
        al = [k * (1 + Z / b) for k, b in zip(w, e)]
        W0 = v[2] + 0.5 * eta * (al[0] * D[0] + al[1] * D[1] + al[2] * D[2]) / (al[0] + al[1] + al[2])
        _, Wt, Wtt = quartic(v, eta)
        Wn, Wnt, _ = quartic(n, eta)
        slope = lambda f: at(f, 0) + 0.5 * eta * (at(f, 1) - at(f, -1))  # noqa: E731
        yield (W0, Wn, Wt, at("NN", 0), Wnt, Wtt, Lv + eta * Ls, Ls / h, slope("LN"), Rv + eta * Rs, Rs / h,
               slope("RN"))


def _moments(U, V, theta, K, side):
    if side == 0:
        u = [torch.ones_like(U), U]
    else:
        s = U / torch.sqrt(2.0 * theta)
        u0 = 0.5 * torch.special.erfc(-side * s)
        u = [u0, U * u0 + side * torch.exp(-s * s) * torch.sqrt(theta / (2.0 * math.pi))]
    v = [torch.ones_like(U), V]
    for k in range(5):
        u.append(U * u[-1] + (k + 1) * theta * u[-2])
        if k < 4:
            v.append(V * v[-1] + (k + 1) * theta * v[-2])
    return u, v, [1.0, K * theta, K * (K + 2) * theta * theta]


_PSI = [[(1.0, 0, 0, 0)], [(1.0, 1, 0, 0)], [(1.0, 0, 1, 0)], [(0.5, 2, 0, 0), (0.5, 0, 2, 0), (0.5, 0, 0, 1)]]


def _psi(mom, A, B=0, coef=None):
    """<u^A v^B psi> or, with coefficients a, <u^A v^B (a . psi) psi>."""
    u, v, x = mom
    out = []
    for k in range(4):
        acc = 0.0
        for c, i, j, m in _PSI[k]:
            if coef is None:
                acc = acc + c * u[A + i] * v[B + j] * x[m]
            else:
                for l in range(4):
                    inner = 0.0
                    for c2, i2, j2, m2 in _PSI[l]:
                        inner = inner + c2 * u[A + i + i2] * v[B + j + j2] * x[m + m2]
                    acc = acc + c * coef[l] * inner
        out.append(acc)
    return torch.stack(out)


def _slope(b, U, V, theta, K):
    Bm = U * U + V * V + (K + 2) * theta
    R4, R3, R2 = 2 * b[3] - Bm * b[0], b[2] - V * b[0], b[1] - U * b[0]
    a3 = (R4 - 2 * U * R2 - 2 * V * R3) / (theta * theta * (K + 2))
    a2, a1 = R3 / theta - V * a3, R2 / theta - U * a3
    return [b[0] - U * a1 - V * a2 - 0.5 * Bm * a3, a1, a2, a3]


def _prim(W):
    U, V = W[1] / W[0], W[2] / W[0]
    p = (GAMMA - 1) * (W[3] - 0.5 * (W[1] * U + W[2] * V))
    return U, V, p, p / W[0]


def _jet_mul(a, b):
    """Product of second-order Taylor jets keyed by (x, y, t) derivative counts."""
    out = {}
    for k in _ORDERS:
        acc = 0.0
        for i, x in a.items():
            j = tuple(p - q for p, q in zip(k, i))
            if min(j) >= 0 and j in b:
                acc = acc + math.prod(math.comb(p, q) for p, q in zip(k, i)) * x * b[j]
        out[k] = acc
    return out


_ORDERS = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (2, 0, 0), (1, 1, 0), (0, 2, 0), (0, 0, 1), (1, 0, 1), (0, 1, 1), (0, 0, 2)]


def _euler(W, Wx, Wy, Wxx, Wxy, Wyy):
    """W_t, W_tt and F_t of the Euler equations (conservative form, Taylor jets)."""
    jets = [{(0, 0, 0): W[k], (1, 0, 0): Wx[k], (0, 1, 0): Wy[k], (2, 0, 0): Wxx[k], (1, 1, 0): Wxy[k],
             (0, 2, 0): Wyy[k]} for k in range(4)]

    def fluxes():
        r = jets[0]
        inv = {(0, 0, 0): 1.0 / r[(0, 0, 0)]}
        for k in _ORDERS[1:]:                      # (rho / rho)_k = 0
            if k not in r:
                continue
            acc = 0.0
            for i in r:
                j = tuple(p - q for p, q in zip(k, i))
                if i != (0, 0, 0) and min(j) >= 0 and j in inv:
                    acc = acc + math.prod(math.comb(p, q) for p, q in zip(k, i)) * r[i] * inv[j]
            inv[k] = -acc * inv[(0, 0, 0)]
        keep = lambda q: {k: x for k, x in q.items() if k in r}  # noqa: E731
        U, V = keep(_jet_mul(jets[1], inv)), keep(_jet_mul(jets[2], inv))
        mU, mV, nV = (keep(_jet_mul(a, b)) for a, b in ((jets[1], U), (jets[1], V), (jets[2], V)))
        p = {k: (GAMMA - 1) * (jets[3][k] - 0.5 * (mU[k] + nV[k])) for k in r}
        H = {k: jets[3][k] + p[k] for k in r}
        UH, VH = keep(_jet_mul(U, H)), keep(_jet_mul(V, H))
        F = [jets[1], {k: mU[k] + p[k] for k in r}, mV, UH]
        G = [jets[2], mV, {k: nV[k] + p[k] for k in r}, VH]
        return F, G, U, V, p

    F, G, U, V, p = fluxes()
    for key, fx, gy in (((0, 0, 1), (1, 0, 0), (0, 1, 0)), ((1, 0, 1), (2, 0, 0), (1, 1, 0)),
                        ((0, 1, 1), (1, 1, 0), (0, 2, 0))):
        for k in range(4):
            jets[k][key] = -(F[k][fx] + G[k][gy])
    F, G, U, V, p = fluxes()
    Wt = torch.stack([j[(0, 0, 1)] for j in jets])
    Ft = torch.stack([f[(0, 0, 1)] for f in F])
    Wtt = torch.stack([-(F[k][(1, 0, 1)] + G[k][(0, 1, 1)]) for k in range(4)])
    return torch.stack([f[(0, 0, 0)] for f in F]), Ft, Wt, Wtt


def _point(pt, kw, dt, stage):
    W0, Wn, Wt, Wnn, Wnt, Wtt, Wl, Wlt, Wln, Wr, Wrt, Wrn = pt
    K = (4 - 2 * GAMMA) / (GAMMA - 1)
    U, V, p, th = _prim(W0)
    F, Ft, W_t, W_tt = _euler(W0, Wn, Wt, Wnn, Wnt, Wtt)
    Ul, Vl, pl, thl = _prim(Wl)
    Ur, Vr, pr, thr = _prim(Wr)
    tau = kw["c_tau"] * dt * ((pl - pr) / (pl + pr)).abs() + (kw["mu"] / p if kw["mu"] > 0 else kw["eps_tau"] * dt)
    h = torch.where(tau > 0, torch.exp(-0.5 * dt / tau.clamp_min(1e-300)), torch.zeros_like(tau))
    ml, mr = _moments(Ul, Vl, thl, K, 1), _moments(Ur, Vr, thr, K, -1)
    sl = (_slope(Wln, Ul, Vl, thl, K), _slope(Wlt, Ul, Vl, thl, K))
    sr = (_slope(Wrn, Ur, Vr, thr, K), _slope(Wrt, Ur, Vr, thr, K))
    Fh = Wl[0] * _psi(ml, 1) + Wr[0] * _psi(mr, 1)
    Th = _psi(ml, 2, 0, sl[0]) + _psi(ml, 1, 1, sl[1]) + _psi(mr, 2, 0, sr[0]) + _psi(mr, 1, 1, sr[1])
    Wh = Wl[0] * _psi(ml, 0) + Wr[0] * _psi(mr, 0)
    Ws = _psi(ml, 1, 0, sl[0]) + _psi(ml, 0, 1, sl[1]) + _psi(mr, 1, 0, sr[0]) + _psi(mr, 0, 1, sr[1])
    del ml, mr, sl, sr
    # rho <(a_n u + a_t v) u psi> of the equilibrium state, whole line
    m0 = _moments(U, V, th, K, 0)
    T0 = _psi(m0, 2, 0, _slope(Wn, U, V, th, K)) + _psi(m0, 1, 1, _slope(Wt, U, V, th, K))
    del m0
    # time integrals over [0, dt/2] and [0, dt] of the second-order flux, as F + t F_t
    q = 4 * tau * (1 - h) / dt ** 2
    dFh, dTh = Fh - F, T0 - Th
    Ftl = Ft - q * (1 - h) * dFh + q * (dt * h - tau * (1 - h)) * dTh
    if stage == 2:
        return Ftl, W_tt
    tat = tau * (1 - h) * (3 - h)
    NS = T0 + Ft
    Fbl = F + tat / dt * dFh - tau * NS + tau / dt * (tat - dt * h * (2 - h)) * dTh
    out = []
    for t, w, c in ((0.5 * dt, h, dt * dt / 8), (dt, h * h, dt * dt / 6)):
        out.append(W0 + t * W_t + c * W_tt + w * (Wh - t * Ws - W0 - t * W_t))
    return Fbl, Ftl, out[0], out[1]


def _faces(Q, S, T, kw, hn, ht, dt, stage):
    """Face results of one orientation: Q, S (4, T + 4, N + 4) face-frame values and h * normal slopes."""
    N = Q.shape[2] - 4
    q = [Q[:, :, o: o + N + 1] for o in range(4)]
    s = [S[:, :, o: o + N + 1] for o in range(4)]
    v, n, nn = _linear(q, s, kw["order"])
    pair = (_char_pair if kw["recon_vars"] else _weno_pair)(q, s, kw["order"], kw["weno_eps"])
    rec = dict(V=v, N=n / hn, NN=nn / hn ** 2, L=pair[0], LN=pair[1] / hn, R=pair[2], RN=pair[3] / hn)
    acc = None
    for pt in _along(rec, T, kw, ht):
        r = _point(pt, kw, dt, stage)
        if stage == 1:
            Fb, Ft, Wm, Wb = r
            r = (0.25 * dt * Fb + dt * dt / 16 * Ft, 0.5 * dt * Fb + dt * dt / 12 * Ft, 0.5 * Wm, 0.5 * Wb)
        else:
            r = tuple(dt * dt / 6 * x for x in r)
        acc = r if acc is None else tuple(a + b for a, b in zip(acc, r))
    return acc


def _ghost(W, kw):
    """Two ghost layers, x sides first, then y."""
    infl = torch.tensor([[r, r * u, r * v, p / (GAMMA - 1) + 0.5 * r * (u * u + v * v)]
                         for r, u, v, p in kw["inflow"]], dtype=torch.float64, device=W.device)
    for ax, odd, lo, normal in ((2, (1, 4, 6, 7, 9), 0, slice(4, 8)), (1, (2, 6, 8, 9, 11), 2, slice(8, 12))):
        n = W.shape[ax]
        sides = []
        for side in (0, 1):
            bc = kw["bc"][lo + side]
            d = [-2, -1] if side == 0 else [n, n + 1]
            if bc == PERIODIC:
                g = W.index_select(ax, torch.tensor([i % n for i in d], device=W.device)).clone()
            elif bc == REFLECT:
                g = W.index_select(ax, torch.tensor([-1 - i if side == 0 else 2 * n - 1 - i for i in d], device=W.device)).clone()
                g[list(odd)] *= -1.0
            else:
                g = W.index_select(ax, torch.tensor([0 if side == 0 else n - 1] * 2, device=W.device)).clone()
                if bc == OUTFLOW:
                    g[normal] = 0.0
                else:
                    g[:4] = infl[lo + side].reshape(4, 1, 1)
                    g[4:] = 0.0
            sides.append(g)
        W = torch.cat([sides[0], W, sides[1]], dim=ax)
    return W


def _stage(W, kw, dx, dy, dt, stage):
    ny, nx = W.shape[1:]
    G = _ghost(W, kw)
    swap = [0, 2, 1, 3]
    fx = _faces(G[:4], dx * G[4:8], ny, kw, dx, dy, dt, stage)
    if kw["dim"] == 1:
        fy = [torch.zeros(4, ny + 1, nx, dtype=W.dtype, device=W.device) for _ in fx]
    else:
        Gy = G.transpose(1, 2)
        fy = [f[swap].transpose(1, 2) for f in _faces(Gy[:4][swap], dy * Gy[8:][swap], nx, kw, dy, dx, dt, stage)]
    return [((a[:, :, 1:] - a[:, :, :-1]) / dx, (b[:, 1:] - b[:, :-1]) / dy) for a, b in zip(fx, fy)]


def _solve(kw, W, steps):
    kw = dict(dict(eps_tau=0.01, c_tau=1.0, weno_eps=1e-6, mu=0.0), **kw)
    dx = (kw["x1"] - kw["x0"]) / kw["nx"]
    dy = (kw["y1"] - kw["y0"]) / kw["ny"] if kw["dim"] == 2 else 1.0
    t = 0.0
    for _ in range(steps):
        U, V, p, _ = _prim(W)
        c, nu2 = torch.sqrt(GAMMA * p / W[0]), 2.0 * kw["mu"] / W[0]
        bound = dx / (U.abs() + c + nu2 / dx)
        if kw["dim"] == 2:
            bound = torch.minimum(bound, dy / (V.abs() + c + nu2 / dy))
        dt = kw["cfl"] * float(bound.min())
        (ax, ay), (bx, by), (mx, my), (ex, ey) = _stage(W, kw, dx, dy, dt, 1)
        star = torch.cat([W[:4] - ax - ay, mx, my])
        R = torch.cat([W[:4] - bx - by, ex, ey])
        (fx, fy), (wx, wy) = _stage(star, kw, dx, dy, dt, 2)
        W = torch.cat([R[:4] - fx - fy, R[4:8] + wx, R[8:] + wy])
        t += dt
    return W, t


def exact(case, seed):
    if case["kind"] == "batch1d" and case["count"] > 40:
        return None                          # hundreds of tiny solves: minutes in plain torch
    rng = np.random.default_rng(seed)
    planes, times = [], []
    for c in _members(case, seed):
        kw, W = _setup(c, rng)
        W, t = _solve(kw, W, case["steps"])
        planes.append(W[[0, 1, 3, 4, 5, 7], 0] if kw["dim"] == 1 else W)
        times.append(t)
    if len(planes) > 1:
        return [torch.cat([w.flatten() for w in planes]), np.array(times)]
    return [planes[0], times[0]]
