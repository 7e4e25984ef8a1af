"""Performance cases of the ADER-SHWENO library: what its users run, through its public entry points.

A case is a dict of plain values.  kind "run" marches a problem to an end time, "advance" takes a
number of CFL steps (the throughput path), "batch" advances many handles together and "train" is
one training step of the flag network.  listed() names the standing cases, draw() makes more of
the same ranges, prepare() builds what a program holds before the call (device arrays, handles),
run() is one pass, work() its unavoidable bytes and operations, exact() the same result from a
plain float64 torch evaluation of the scheme that shares no code with the library.
"""
import math
import random

import numpy as np
import torch

from paper_2304_09724_gb300 import flagnet
from paper_2304_09724_gb300 import shweno as S

GAMMA = 1.4
PERIODIC, OUTFLOW, REFLECTIVE, INFLOW, DMR_BOTTOM, DMR_TOP = range(6)
POST = (8.0, 57.1597, -33.0012, 563.544)
FIRST = 4  # problems of a batch that are returned one by one (and have an exact result)


def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


# ------------------------------------------------------------------------------------ the cases
def _solve(name, flow, nx, ny=1, weights="plain", charwise=False, quintic=False, **more):
    return dict(name=name, flow=flow, nx=nx, ny=ny, weights=weights, charwise=charwise, quintic=quintic, **more)


def listed():
    return [
        # a small scalar problem marched to its end time: the latency of a whole short run
        _solve("burgers1d_run_200", "burgers_sine", 200, kind="run", t_final=0.5 / math.pi),
        # a shock tube at the usual resolution, marched to its end time on outflow sides
        _solve("lax1d_run_200", "lax", 200, kind="run", t_final=1.3),
        # a large 1D mesh (the 1D throughput workload's size)
        _solve("euler1d_4m", "wave1d", 1 << 22, kind="advance", steps=2),
        # the coarse end of a refinement study: a mesh far smaller than the GPU
        _solve("vortex_40", "vortex", 40, 40, kind="advance", steps=12),
        # the four-shock quadrant problem at its published mesh, nonlinear weights at work everywhere
        _solve("quadrants_400", "quadrants", 400, 400, kind="advance", steps=2),
        # the double Mach reflection with the learned flag, walls and imposed states, a wide mesh
        _solve("dmr_1024x256_learned", "dmr", 1024, 256, weights="learned", kind="advance", steps=2),
        # the headline mesh, one step
        _solve("vortex_2048", "vortex", 2048, 2048, kind="advance", steps=1),
        # the 2D scalar law on an odd, ragged mesh
        _solve("burgers2d_501x387", "burgers2d", 501, 387, kind="advance", steps=4),
        # the characteristic-wise option at the finest mesh of the published vortex table but one
        _solve("vortex_160_charwise", "vortex", 160, 160, charwise=True, kind="advance", steps=4),
        # an ensemble of 1D Riemann problems of uneven sizes in one batch
        dict(name="batch1d_64", kind="batch", flow="riemann1d", problems=64, nmin=400, nmax=16384, steps=16),
        # an ensemble of 2D quadrant problems of uneven sizes in one batch
        dict(name="batch2d_6", kind="batch", flow="quadrants", problems=6, nmin=128, nmax=448, steps=2),
        # one training step of the flag network (forward, backward, optimiser) at its batch size
        dict(name="flagnet_train_16384", kind="train", samples=16384),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    pick = rng.random()
    if pick < 0.14:
        flow, t = rng.choice([("burgers_sine", 0.5 / math.pi), ("lax", 1.3), ("wave1d", 0.5), ("shu_osher", 0.4)])
        n = _log_int(rng, 40, 800)
        return _pure(_solve("", flow, n, kind="run", t_final=round(t * rng.uniform(0.5, 1.0), 6),
                            charwise=flow == "lax" and rng.random() < 0.3, quintic=flow == "wave1d" and rng.random() < 0.3))
    if pick < 0.28:
        flow = rng.choice(["wave1d", "burgers_sine", "shu_osher"])
        return _pure(_solve("", flow, _log_int(rng, 1000, 1 << 22), kind="advance", steps=rng.randint(1, 4)))
    if pick < 0.74:
        flow = rng.choice(["vortex", "vortex", "smooth2d", "quadrants", "quadrants", "dmr", "burgers2d"])
        n = _log_int(rng, 20, 1400)
        nx, ny = n, n
        if flow == "dmr":
            nx, ny = 4 * max(16, n // 2), max(16, n // 2)
        elif flow in ("smooth2d", "burgers2d"):
            ny = max(8, int(n * rng.uniform(0.3, 1.0)))
        weights = rng.choice(["plain", "plain", "linear", "learned"]) if flow in ("vortex", "smooth2d") else \
            (rng.choice(["plain", "learned"]) if flow == "dmr" else "plain")
        option = rng.random()
        smooth = flow in ("vortex", "smooth2d") and weights == "plain"
        return _pure(_solve("", flow, nx, ny, weights=weights, kind="advance", steps=rng.randint(1, 4) if n < 700 else 1,
                            charwise=smooth and option < 0.2, quintic=smooth and 0.2 <= option < 0.35))
    if pick < 0.84:
        return dict(kind="batch", flow="riemann1d", problems=_log_int(rng, 8, 128), nmin=400, nmax=_log_int(rng, 2000, 16384),
                    steps=rng.randint(4, 16))
    if pick < 0.92:
        return dict(kind="batch", flow="quadrants", problems=rng.randint(2, 12), nmin=64, nmax=_log_int(rng, 100, 448),
                    steps=rng.randint(1, 2))
    return dict(kind="train", samples=_log_int(rng, 1000, 65536))


def _pure(case):
    case.pop("name")
    return case


# ------------------------------------------------------------------------------------ initial data
def _euler(rho, u, p, v=None):
    """Conserved state of primitive tensors (1D: no v)."""
    one = rho + 0.0 * u
    if v is None:
        return torch.stack([one, rho * u, p / (GAMMA - 1.0) + 0.5 * rho * u * u + 0.0 * one])
    z = 0.0 * one + 0.0 * v
    return torch.stack([one + z, rho * u + z, rho * v + z, p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v) + z])


def _flow(flow, seed):
    """(function of x (, y) giving the conserved state, domain, sides, inflow states) of a seeded problem."""
    r = random.Random(seed * 1000003 + sum(map(ord, flow)))
    U = r.uniform
    tau = 2.0 * math.pi
    none = [[0.0] * 4 for _ in range(4)]
    if flow == "burgers_sine":  # a sine that steepens, periodic
        a, ph = U(0.85, 1.1), U(0, tau)
        return lambda x: (0.5 + a * torch.sin(math.pi * x + ph))[None], (0.0, 2.0, 0.0, 1.0), (0, 0, 0, 0), none
    if flow == "wave1d":  # a smooth wave in all three fields, periodic
        a, ph = [U(0.05, 0.2) for _ in range(3)], [U(0, tau) for _ in range(3)]
        return (lambda x: _euler(1.0 + a[0] * torch.sin(math.pi * x + ph[0]), 1.0 + a[1] * torch.sin(math.pi * x + ph[1]),
                                 1.0 + a[2] * torch.sin(tau * x + ph[2]))), (0.0, 2.0, 0.0, 1.0), (0, 0, 0, 0), none
    if flow == "lax":  # the Lax shock tube's two states, a little varied
        k = [U(0.95, 1.05) for _ in range(6)]
        L, R = (0.445 * k[0], 0.698 * k[1], 3.528 * k[2]), (0.5 * k[3], 0.0, 0.571 * k[4])
        return (lambda x: _two(x, 0.0, L, R)), (-5.0, 5.0, 0.0, 1.0), (OUTFLOW, OUTFLOW, 0, 0), none
    if flow == "riemann1d":  # a random Riemann problem
        L, R = [(U(0.2, 2.0), U(-0.7, 0.7), U(0.3, 10.0)) for _ in range(2)]
        return (lambda x: _two(x, 0.5, L, R)), (0.0, 1.0, 0.0, 1.0), (OUTFLOW, OUTFLOW, 0, 0), none
    if flow == "shu_osher":  # a Mach 3 shock entering a density wave
        a, k, ph = U(0.15, 0.25), U(4.0, 6.0), U(0, tau)

        def f(x):
            left = x < -4.0
            w = lambda p, q: torch.where(left, torch.full_like(x, p), q if torch.is_tensor(q) else torch.full_like(x, q))
            return _euler(w(3.857143, 1.0 + a * torch.sin(k * x + ph)), w(2.629369, 0.0), w(10.333333, 1.0))
        return f, (-5.0, 5.0, 0.0, 1.0), (OUTFLOW, OUTFLOW, 0, 0), none
    if flow == "vortex":  # an isentropic vortex in a uniform stream, periodic
        s, cx, cy = U(4.5, 5.5), U(3.0, 7.0), U(3.0, 7.0)

        def f(x, y):
            xr, yr = torch.remainder(x - cx + 5.0, 10.0) - 5.0, torch.remainder(y - cy + 5.0, 10.0) - 5.0
            e = math.exp(0.5) * torch.exp(-0.5 * xr * xr) * torch.exp(-0.5 * yr * yr)
            base = 1.0 - (GAMMA - 1.0) * s * s / (8.0 * GAMMA * math.pi ** 2) * e * e
            rho = base * base * torch.sqrt(base)
            return _euler(rho, 1.0 - s / tau * e * yr, rho * base, 1.0 + s / tau * e * xr)
        return f, (0.0, 10.0, 0.0, 10.0), (0, 0, 0, 0), none
    if flow == "smooth2d":  # smooth waves in every field, periodic
        k = [(r.randint(1, 2), r.randint(0, 2), U(0, tau), U(-0.1, 0.1)) for _ in range(4)]

        def f(x, y):
            m = [a * torch.sin(tau * (kx * x + ky * y) + ph) for kx, ky, ph, a in k]
            return _euler(1.0 + m[0], 0.4 + m[1], 1.0 + m[2], -0.3 + m[3])
        return f, (0.0, 1.0, 0.0, 1.0), (0, 0, 0, 0), none
    if flow == "quadrants":  # the four-shock quadrant problem, its states a little varied
        k = [[1.0 + U(-0.03, 0.03) for _ in range(4)] for _ in range(4)]
        q = [(1.1, 0.0, 0.0, 1.1), (0.5065, 0.8939, 0.0, 0.35), (1.1, 0.8939, 0.8939, 1.1), (0.5065, 0.0, 0.8939, 0.35)]
        q = [tuple(a * b for a, b in zip(p, kk)) for p, kk in zip(q, k)]

        def f(x, y):
            e, n = (x >= 0.5) & (y > -1.0), (y >= 0.5) & (x > -1.0)
            at = lambda c: torch.where(n, torch.where(e, q[0][c], q[1][c]), torch.where(e, q[3][c], q[2][c])).to(torch.float64)
            return _euler(at(0), at(1), at(3), at(2))
        return f, (0.0, 1.0, 0.0, 1.0), (OUTFLOW,) * 4, none
    if flow == "dmr":  # the double Mach reflection; the gas ahead of the shock carries a weak density wave
        a, kx, ph = U(0.005, 0.02), r.randint(1, 4), U(0, tau)

        def f(x, y):
            post = y >= math.sqrt(3.0) * (x - 1.0 / 6.0)
            rho = 1.4 * (1.0 + a * torch.sin(math.pi * kx * x + ph)) + 0.0 * y
            return torch.stack([torch.where(post, POST[0], rho), torch.where(post, POST[1], 0.0 * rho),
                                torch.where(post, POST[2], 0.0 * rho), torch.where(post, POST[3], 2.5 + 0.0 * rho)])
        return f, (0.0, 4.0, 0.0, 1.0), (INFLOW, OUTFLOW, DMR_BOTTOM, DMR_TOP), [list(POST)] + none[1:]
    if flow == "burgers2d":  # a diagonal wave of the 2D scalar law that changes sign, periodic
        a, ph = U(0.8, 1.1), U(0, tau)
        return lambda x, y: (0.3 + a * torch.sin(math.pi * (x + y) + ph))[None], (0.0, 2.0, 0.0, 2.0), (0, 0, 0, 0), none
    raise ValueError(flow)


def _two(x, xs, L, R):
    w = lambda c: torch.where(x < xs, torch.full_like(x, L[c]), torch.full_like(x, R[c]))
    return _euler(w(0), w(1), w(2))


def _initial(flow, nx, ny, seed):
    """Cell averages and derivative averages (Gauss rules; derivatives from edge values taken just
    inside the cell) of a seeded problem: dict of float64 tensors on the device."""
    f, dom, _, _ = _flow(flow, seed)
    pts, wts = (0.5 * v for v in np.polynomial.legendre.leggauss(4))
    D, kw = _dev(), dict(dtype=torch.float64)
    dx, dy = (dom[1] - dom[0]) / nx, (dom[3] - dom[2]) / ny
    x = dom[0] + (torch.arange(nx, device=D, **kw) + 0.5) * dx
    h = 0.5 - 1e-9
    if flow in ("burgers_sine", "wave1d", "lax", "riemann1d", "shu_osher"):
        W = sum(w * f(x + s * dx) for s, w in zip(pts, wts))
        st = {"W": W, "V": (f(x + h * dx) - f(x - h * dx)) / dx}
        return {k: v.contiguous() for k, v in st.items()}
    x, y = x[None, :], (dom[2] + (torch.arange(ny, device=D, **kw) + 0.5) * dy)[:, None]
    W = V = Y = 0.0
    for s, w in zip(pts, wts):
        for s2, w2 in zip(pts, wts):
            W = W + w * w2 * f(x + s * dx, y + s2 * dy)
        V = V + w * (f(x + h * dx, y + s * dy) - f(x - h * dx, y + s * dy)) / dx
        Y = Y + w * (f(x + s * dx, y + h * dy) - f(x + s * dx, y - h * dy)) / dy
    c = [f(x + a * h * dx, y + b * h * dy) for a, b in ((1, 1), (-1, 1), (1, -1), (-1, -1))]
    Z = (c[0] - c[1] - c[2] + c[3]) / (dx * dy)
    full = (W.shape[0], ny, nx)
    return {k: v.expand(full).contiguous() for k, v in (("W", W), ("V", V), ("Y", Y), ("Z", Z))}


def _eq(flow):
    return S.BURGERS if flow.startswith("burgers") else S.EULER


def _dim(flow):
    return 2 if flow in ("vortex", "smooth2d", "quadrants", "dmr", "burgers2d") else 1


# ------------------------------------------------------------------------------------ one pass
def _handle(flow, nx, ny, seed, weights="plain", charwise=False, quintic=False):
    _, dom, bc, inflow = _flow(flow, seed)
    mode = {"plain": 0, "linear": 1, "learned": 2}[weights]
    sol = S.Solver(_dim(flow), _eq(flow), nx, ny, dom, bc, inflow=inflow, flag_mode=mode, charwise=charwise, quintic=quintic)
    if weights == "learned":
        params, thr = flagnet.load()
        S.shweno_set_flag_net(sol.h, params, thr)
    init = _initial(flow, nx, ny, seed)
    return {"sol": sol, "init": init, "out": {k: torch.empty_like(v) for k, v in init.items()}}


def _sizes(case):
    """Side lengths of a batch's problems, spread over [nmin, nmax] (even sides in 2D)."""
    r = random.Random(7 * case["problems"] + case["nmax"])
    n = [r.randint(case["nmin"], case["nmax"]) for _ in range(case["problems"])]
    return n if _dim(case["flow"]) == 1 else [v - v % 2 for v in n]


def _net_start(case, seed):
    """A labelled sample batch and the network and optimiser state in the middle of a training run."""
    D, n = _dev(), case["samples"]
    g = torch.Generator(device="cpu").manual_seed(seed)
    k = S.FLAG_PARAMS
    x = torch.randn(n, S.FLAG_FEATURES, generator=g) * 0.5
    y = (x[:, 0] + 0.3 * torch.randn(n, generator=g) > 0.8).float()
    params = torch.from_numpy(flagnet.init_params(seed)) + 0.02 * torch.randn(k, generator=g)
    m, v = 1e-3 * torch.randn(k, generator=g), 1e-4 * (0.5 + torch.rand(k, generator=g))
    return [t.to(D).contiguous() for t in (x, y, params, m, v)]


def prepare(case, seed):
    if case["kind"] == "train":
        x, y, params, m, v = _net_start(case, seed)
        return {"case": case, "x": x, "y": y, "params": params, "m": m, "v": v, "step": 20,
                "grad": torch.zeros_like(params), "loss": torch.zeros(1, device=x.device)}
    if case["kind"] == "batch":
        ps = [_handle(case["flow"], n, n, 1000 * seed + i) for i, n in enumerate(_sizes(case))]
        rest = {}  # the results of all problems but the first few lie in one array per field
        for k in ps[0]["out"]:
            rest[k] = torch.empty(sum(p["out"][k].numel() for p in ps[FIRST:]), dtype=torch.float64, device=_dev())
            parts = rest[k].split([p["out"][k].numel() for p in ps[FIRST:]]) if len(ps) > FIRST else []
            for p, part in zip(ps[FIRST:], parts):
                p["out"][k] = part.view(p["out"][k].shape)
        return {"case": case, "problems": ps, "batch": S.Batch([p["sol"] for p in ps]), "rest": rest}
    h = _handle(case["flow"], case["nx"], case["ny"], seed, case["weights"], case["charwise"], case["quintic"])
    return {"case": case, **h}


def _read(p):
    o = p["out"]
    S.shweno_get_state(p["sol"].h, o["W"], o["V"], o.get("Y"), o.get("Z"))
    return o


def run(state):
    case = state["case"]
    if case["kind"] == "train":
        state["step"] += 1
        S.shweno_mlp_grad(state["params"], state["x"], state["y"], 4.0, state["grad"], state["loss"])
        S.shweno_mlp_adam(state["params"], state["grad"], state["m"], state["v"], state["step"], 2e-3)
        return [state[k] for k in ("loss", "grad", "params", "m", "v")]
    if case["kind"] == "batch":
        for p in state["problems"]:
            p["sol"].set_state(p["init"])
        _, status = state["batch"].run(1e9, 0.6, max_steps=case["steps"])
        return [np.array(status), [_read(p) for p in state["problems"]][:FIRST], state["rest"]]
    sol = state["sol"]
    sol.set_state(state["init"])
    if case["kind"] == "run":
        t, n = sol.run(case["t_final"], 0.6)
        return [_read(state), t, n]
    S.shweno_advance(sol.h, case["steps"], 0.6)
    return [_read(state)]


# ------------------------------------------------------------------------------------ its work
def work(case):
    """Bytes: the state read and written once a step, in float64.  Operations of the method per
    cell and step (a fused multiply-add counts two): in 2D Euler 4 x-face points (3 Gauss points
    and a corner) of 5025, 3 y-face points of 4995 and 16 first-pass reconstructions; the others
    counted alike."""
    if case["kind"] == "train":
        n, k = case["samples"], S.FLAG_PARAMS
        return {"bytes": 4.0 * (n * (S.FLAG_FEATURES + 1) + 7 * k), "flops": 6.0 * n * k}
    per = {(1, S.BURGERS): 260.0, (1, S.EULER): 1150.0, (2, S.BURGERS): 5000.0, (2, S.EULER): 36500.0}
    dim, eq = _dim(case["flow"]), _eq(case["flow"])
    nc = 1 if eq == S.BURGERS else dim + 2
    if case["kind"] == "batch":
        cells = sum(n ** dim for n in _sizes(case)) * case["steps"]
    elif case["kind"] == "run":
        dom = _flow(case["flow"], 0)[1]
        speed = {"burgers_sine": 1.5, "lax": 4.7, "wave1d": 2.4, "shu_osher": 4.7}[case["flow"]]
        cells = case["nx"] * max(1.0, case["t_final"] * speed * case["nx"] / (0.6 * (dom[1] - dom[0])))
    else:
        cells = case["nx"] * case["ny"] * case["steps"]
    return {"bytes": cells * 2.0 * 8.0 * nc * 2 ** dim, "flops": cells * per[dim, eq]}


# ------------------------------------------------------------------------------------ float64 reference
# The scheme evaluated plainly: reconstruction polynomials from small linear systems, smoothness
# integrals as quadratic forms, eigenvector matrices, dense series products.
def _moments(deg, c):
    """Average of xi^k over the cell centred at c (width 1), k = 0..deg."""
    return [((c + 0.5) ** (k + 1) - (c - 0.5) ** (k + 1)) / (k + 1) for k in range(deg + 1)]


def _slopes(deg, c):
    return [(c + 0.5) ** k - (c - 0.5) ** k for k in range(deg + 1)]


def _tables(quintic):
    deg = 5 if quintic else 4
    rows = [_moments(deg, c) for c in (-1, 0, 1)] + [_slopes(deg, c) for c in ((-1, 0, 1) if quintic else (-1, 1))]
    fit = np.linalg.inv(np.array(rows))  # (W-, W0, W+, v-, (v0,) v+) -> monomial coefficients
    beta = np.zeros((deg + 1, deg + 1))
    for a in range(1, deg + 1):  # sum over a of the integral of (d^a p)^2
        for i in range(a, deg + 1):
            for j in range(a, deg + 1):
                m = i + j - 2 * a
                beta[i, j] += math.perm(i, a) * math.perm(j, a) * ((0.5 ** (m + 1) - (-0.5) ** (m + 1)) / (m + 1))
    return deg, fit, beta


def _poly(T, d):
    """p1's monomial coefficients from the stencil data d (list of tensors)."""
    return [sum(float(c) * v for c, v in zip(row, d)) for row in T[1]]


def _weights(T, c, Wm, W0, Wp, flag):
    """(A, B, C): p = A p1 + B p2 + C p3; linear weights where flag is 0."""
    deg, _, beta = T
    b1 = sum(float(beta[i, j]) * c[i] * c[j] for i in range(1, deg + 1) for j in range(1, deg + 1) if beta[i, j])
    b2, b3 = (W0 - Wm) ** 2, (Wp - W0) ** 2
    tau = (0.5 * ((b1 - b2).abs() + (b1 - b3).abs())) ** 2
    g = (0.994, 0.003, 0.003)
    w = [gl * (1.0 + tau / (b + 1e-6)) for gl, b in zip(g, (b1, b2, b3))]
    s = w[0] + w[1] + w[2]
    A = w[0] / s / g[0]
    B, C = w[1] / s - A * g[1], w[2] / s - A * g[2]
    if flag is True:
        return A, B, C
    return torch.where(flag, A, 1.0), torch.where(flag, B, 0.0), torch.where(flag, C, 0.0)


def _combine(T, mix, d):
    """Monomial coefficients of A p1 + B p2 + C p3 for stencil data d."""
    c = _poly(T, d)
    A, B, C = mix
    e = [A * v for v in c]
    e[0] = e[0] + (B + C) * d[1]
    e[1] = e[1] + B * (d[1] - d[0]) + C * (d[2] - d[1])
    return e


def _shift(e, x):
    """Taylor coefficients 0..4 about x."""
    return [sum(math.comb(j, k) * x ** (j - k) * e[j] for j in range(k, len(e))) for k in range(5)]


def _stencil(T, W, v, c0, n, axis):
    """Stencil data of n cells along axis, the first one's left neighbour at index c0."""
    at = lambda a, k: a.narrow(axis, c0 + k, n)
    vs = (0, 1, 2) if T[0] == 5 else (0, 2)
    return [at(W, k) for k in range(3)] + [at(v, k) for k in vs]


def _prim(W):
    rho, u = W[0], W[1] / W[0]
    v = W[2] / W[0] if len(W) == 4 else 0.0 * u
    p = (GAMMA - 1.0) * (W[-1] - 0.5 * rho * (u * u + v * v))
    return rho, u, v, p, torch.sqrt(GAMMA * p / rho), (W[-1] + p) / rho


def _flux(W):
    """Flux along x."""
    if len(W) == 1:
        return [0.5 * W[0] * W[0]]
    _, u, _, p, _, _ = _prim(W)
    F = [W[1], W[1] * u + p, u * (W[-1] + p)]
    return F if len(W) == 3 else F[:2] + [W[2] * u, F[2]]


def _leading(WL, WR):
    if len(WL) == 1:
        l, r = WL[0], WR[0]
        fan = torch.where(l >= 0, l, torch.where(r <= 0, r, 0.0 * l))
        return [torch.where(l > r, torch.where(0.5 * (l + r) >= 0, l, r), fan)]
    L, R = _prim(WL), _prim(WR)
    SL, SR = torch.minimum(L[1] - L[4], R[1] - R[4]), torch.maximum(L[1] + L[4], R[1] + R[4])
    mL, mR = L[0] * (SL - L[1]), R[0] * (SR - R[1])
    Ss = (R[3] - L[3] + L[1] * mL - R[1] * mR) / (mL - mR)
    left = Ss >= -1e-12 * torch.maximum(L[4], R[4])
    w = lambda a, b: torch.where(left, a, b)
    Sk, un, vn, rho, p, E = w(SL, SR), w(L[1], R[1]), w(L[2], R[2]), w(L[0], R[0]), w(L[3], R[3]), w(WL[-1], WR[-1])
    f = rho * (Sk - un) / (Sk - Ss)
    star = [f, f * Ss, f * (E / rho + (Ss - un) * (Ss + p / (rho * (Sk - un))))]
    if len(WL) == 4:
        star = star[:2] + [f * vn, star[2]]
    return [torch.where(SL >= 0, a, torch.where(SR < 0, b, s)) for a, b, s in zip(WL, WR, star)]


def _eigen(W):
    """Speeds, right eigenvectors (lists) and left eigenvectors of the x-flux Jacobian at W."""
    _, u, v, _, c, H = _prim(W)
    two = len(W) == 4
    b1 = (GAMMA - 1.0) / (c * c)
    q = u * u + v * v
    b2, one, zero = 0.5 * b1 * q, torch.ones_like(u), torch.zeros_like(u)
    cut = lambda r: r if two else [r[0], r[1], r[3]]
    lam, R, L = [], [], []
    for s in (-1.0, 1.0):
        lam.append(u + s * c)
        R.append(cut([one, u + s * c, v, H + s * u * c]))
        L.append(cut([0.5 * (b2 - s * u / c), 0.5 * (s / c - b1 * u), -0.5 * b1 * v, 0.5 * b1]))
    lam.append(u)
    R.append(cut([one, u, v, 0.5 * q]))
    L.append(cut([1.0 - b2, b1 * u, b1 * v, -b1]))
    if two:
        lam.append(u)
        R.append([zero, zero, one, v])
        L.append([-v, zero, one, zero])
    return lam, R, L, c


def _ck(a, eq, lx, ly):
    """Time Taylor coefficients 0..4 at the point from the spatial ones a[q][(m, n)]; lx = 1/dx."""
    two = ly is not None
    nc = len(a)
    Sr = [{(m, n, 0): v for (m, n), v in aq.items()} for aq in a]
    names = ("u", "v", "mu", "mv", "nv", "p", "H", "uH", "vH", "uu")
    X = {k: {} for k in names}

    def mul(A, B, i):
        return sum(A[p, q, t] * B[i[0] - p, i[1] - q, i[2] - t]
                   for p in range(i[0] + 1) for q in range(i[1] + 1) for t in range(i[2] + 1))

    def div(A, Q, i):  # Q rho = A
        r = Sr[0]
        s = A[i]
        for p in range(i[0] + 1):
            for q in range(i[1] + 1):
                for t in range(i[2] + 1):
                    if p + q + t:
                        s = s - r[p, q, t] * Q[i[0] - p, i[1] - q, i[2] - t]
        return s / r[0, 0, 0]

    for k in range(4):
        F, G = [{} for _ in range(nc)], [{} for _ in range(nc)]
        for m in range(5 - k):
            for n in range(5 - k - m if two else 1):
                i = (m, n, k)
                if eq == S.BURGERS:
                    F[0][i] = G[0][i] = 0.5 * mul(Sr[0], Sr[0], i)
                    continue
                E = Sr[-1]
                X["u"][i] = div(Sr[1], X["u"], i)
                X["mu"][i] = mul(Sr[1], X["u"], i)
                kin = X["mu"][i]
                if two:
                    X["v"][i] = div(Sr[2], X["v"], i)
                    X["mv"][i], X["nv"][i] = mul(Sr[1], X["v"], i), mul(Sr[2], X["v"], i)
                    kin = kin + X["nv"][i]
                X["p"][i] = (GAMMA - 1.0) * (E[i] - 0.5 * kin)
                X["H"][i] = E[i] + X["p"][i]
                X["uH"][i] = mul(X["u"], X["H"], i)
                f = [Sr[1][i], X["mu"][i] + X["p"][i], X["uH"][i]]
                if two:
                    X["vH"][i] = mul(X["v"], X["H"], i)
                    f = f[:2] + [X["mv"][i], f[2]]
                    for q, gq in enumerate([Sr[2][i], X["mv"][i], X["nv"][i] + X["p"][i], X["vH"][i]]):
                        G[q][i] = gq
                for q in range(nc):
                    F[q][i] = f[q]
        for q in range(nc):
            for m in range(4 - k):
                for n in range(4 - k - m if two else 1):
                    s = (m + 1) * lx * F[q][m + 1, n, k]
                    if two:
                        s = s + (n + 1) * ly * G[q][m, n + 1, k]
                    Sr[q][m, n, k + 1] = -s / (k + 1)
    return [[Sr[q][0, 0, k] for k in range(5)] for q in range(nc)]


def _sides(T, Ws, Vs, flag, basis, corner_axis):
    """Across-face Taylor coefficients on both sides of the faces: Ws[k], Vs[k] ([nc, .., n + 4]) are
    the stencil data of order k along the face.  Returns left and right [k][m] of [nc, .., n + 1]."""
    ax = corner_axis
    n = Ws[0].shape[ax] - 4
    out = []
    if basis is None:
        d0 = _stencil(T, Ws[0], Vs[0], 0, n + 2, ax)
        mix = _weights(T, _poly(T, d0), d0[0], d0[1], d0[2], flag if flag is True else flag.narrow(ax - 1, 1, n + 2))
        for k in range(len(Ws)):
            e = _combine(T, mix, _stencil(T, Ws[k], Vs[k], 0, n + 2, ax))
            out.append((_shift(e, 0.5)[: 5 - k], _shift(e, -0.5)[: 5 - k]))
        return [[v.narrow(ax, 0, n + 1) for v in l] for l, _ in out], [[v.narrow(ax, 1, n + 1) for v in r] for _, r in out]
    R, L = basis
    proj = lambda M, v: torch.stack([sum(M[f][q] * v[q] for q in range(len(M))) for f in range(len(M))])
    back = lambda v: torch.stack([sum(R[f][q] * v[f] for f in range(len(R))) for q in range(len(R))])
    res = []
    for side, x in ((0, 0.5), (1, -0.5)):
        mix, rows = None, []
        for k in range(len(Ws)):
            d = [proj(L, v) for v in _stencil(T, Ws[k], Vs[k], side, n + 1, ax)]
            if mix is None:
                fl = flag if flag is True else flag.narrow(ax - 1, 1 + side, n + 1)
                mix = _weights(T, _poly(T, d), d[0], d[1], d[2], fl)
            rows.append([back(v) for v in _shift(_combine(T, mix, d), x)[: 5 - k]])
        res.append(rows)
    return res


def _points(left, right, eq, dt, lx, ly):
    """Leading term, derivative problems, time expansion: (time-averaged flux, state at dt, both [nc, ..])."""
    nc = left[0][0].shape[0]
    Ws = _leading(list(left[0][0]), list(right[0][0]))
    if nc > 1:
        lam, R, L, scale = _eigen(Ws)
    else:
        lam, R, L = [Ws[0]], [[torch.ones_like(Ws[0])]], [[torch.ones_like(Ws[0])]]
        scale = torch.maximum(left[0][0][0].abs(), right[0][0][0].abs())
    a = [{} for _ in range(nc)]
    for q in range(nc):
        a[q][0, 0] = Ws[q]
    side = [torch.where(s > 1e-12 * scale, 1.0, torch.where(s < -1e-12 * scale, 0.0, 0.5)) for s in lam]
    for k in range(len(left)):
        for m in range(5 - k):
            if m + k == 0:
                continue
            dl, dr = left[k][m], right[k][m]
            amp = [dr_ + h * (dl_ - dr_) for h, dl_, dr_ in
                   ((side[w], sum(L[w][q] * dl[q] for q in range(nc)), sum(L[w][q] * dr[q] for q in range(nc))) for w in range(len(lam)))]
            for q in range(nc):
                a[q][m, k] = sum(R[w][q] * amp[w] for w in range(len(lam)))
    tc = _ck(a, eq, lx, ly)
    s5 = 0.5 / math.sqrt(5.0)
    F = 0.0
    for node, w in ((0.0, 1 / 12), (0.5 - s5, 5 / 12), (0.5 + s5, 5 / 12), (1.0, 1 / 12)):
        W = [sum(c[k] * (node * dt) ** k for k in range(5)) for c in tc]
        F = F + w * torch.stack(_flux(W))
    return F, torch.stack(W)


def _ghosts(u, field, kinds, ax, fixed, nc, eq):
    """Two ghost layers along axis ax (1: y, 2: x; the last axis in 1D) of field W, V, Y or Z."""
    n = u.shape[ax]
    parts = [None, u, None]
    normal = 1 if ax == u.dim() - 1 else 2
    for side in (0, 1):
        kind = kinds[side]
        if kind == PERIODIC:
            g = u.narrow(ax, n - 2 if side == 0 else 0, 2)
        elif kind == OUTFLOW:
            e = u.narrow(ax, 0 if side == 0 else n - 1, 1)
            g = torch.cat([e, e], ax)
        elif kind in (REFLECTIVE, DMR_BOTTOM):
            g = u.narrow(ax, 0 if side == 0 else n - 2, 2).flip(ax).clone()
            if field in ({1: "VZ", 2: "YZ"}[normal]):
                g = -g
            if eq == S.EULER:
                g[normal] = -g[normal]
        if kind in (INFLOW, DMR_BOTTOM, DMR_TOP):
            g = fixed(side, kind, field, None if kind in (INFLOW, DMR_TOP) else g)
        parts[0 if side == 0 else 2] = g
    return torch.cat(parts, ax)


def _pad(st, dom, bc, inflow, t, eq):
    nc = st["W"].shape[0]
    if st["W"].dim() == 2:
        return {k: _ghosts(v, k, bc[:2], 1, None, nc, eq) for k, v in st.items()}
    ny, nx = st["W"].shape[1:]
    dx, dy = (dom[1] - dom[0]) / nx, (dom[3] - dom[2]) / ny
    kw = dict(dtype=torch.float64, device=st["W"].device)
    post, pre = torch.tensor(POST, **kw)[:, None, None], torch.tensor((1.4, 0.0, 0.0, 2.5), **kw)[:, None, None]
    xc = dom[0] + (torch.arange(-2, nx + 2, **kw) + 0.5)[None, :] * dx

    def along_x(side, kind, field, g):
        v = torch.tensor(inflow[side], **kw)[:nc, None, None].expand(nc, ny, 2)
        return v if field == "W" else 0.0 * v

    def along_y(side, kind, field, g):
        if kind == DMR_BOTTOM:
            imposed = post if field == "W" else 0.0 * post
            return torch.where((xc < 1.0 / 6.0)[None], imposed, g)
        yc = dom[3] + (torch.arange(2, **kw) + 0.5)[:, None] * dy
        past = yc >= math.sqrt(3.0) * (xc - 1.0 / 6.0) - 20.0 * t
        v = torch.where(past[None], post, pre)
        return v if field == "W" else 0.0 * v

    out = {}
    for k, u in st.items():
        u = _ghosts(u, k, bc[:2], 2, along_x, nc, eq)
        u = _ghosts(u, k, bc[2:], 1, along_y, nc, eq)
        if bc[0] == INFLOW:
            u[:, :, :2] = torch.tensor(inflow[0], **kw)[:, None, None] if k == "W" else 0.0
        out[k] = u
    return out


def _pad_flags(raw, bc):
    """Two ghost layers of a cell flag; sides that impose a state count as flagged."""
    for ax, kinds in ((1, bc[:2]), (0, bc[2:])):
        n = raw.shape[ax]
        g = []
        for side in (0, 1):
            if kinds[side] == PERIODIC:
                g.append(raw.narrow(ax, n - 2 if side == 0 else 0, 2))
            elif kinds[side] == OUTFLOW:
                e = raw.narrow(ax, 0 if side == 0 else n - 1, 1)
                g.append(torch.cat([e, e], ax))
            elif kinds[side] == REFLECTIVE:
                g.append(raw.narrow(ax, 0 if side == 0 else n - 2, 2).flip(ax))
            else:
                g.append(torch.ones_like(raw.narrow(ax, 0, 2)))
        raw = torch.cat([g[0], raw, g[1]], ax)
    return raw


def _learned_flags(P, dx, dy, bc):
    """The network on every cell of the padded state P, dilated by one cell, padded."""
    params, thr = flagnet.load()
    w = torch.from_numpy(params).to(P["W"].device).double()
    nin, nh = S.FLAG_FEATURES, 32
    cut = lambda u, j=0, i=0: u[2 + j: u.shape[0] - 2 + j, 2 + i: u.shape[1] - 2 + i]
    feats = []
    for q in (0, 3):
        W = P["W"][q]
        nb = [cut(W, j, i) for j in (-1, 0, 1) for i in (-1, 0, 1)]
        c = nb[4]
        mx, mn = torch.stack(nb).amax(0), torch.stack(nb).amin(0)
        sc = mx - mn + 1e-12 * c.abs() + 1e-300
        feats += [(v - c) / sc for k, v in enumerate(nb) if k != 4]
        feats += [dx * cut(P["V"][q]) / sc, dy * cut(P["Y"][q]) / sc,
                  torch.log10((mx - mn) / (c.abs() + 1e-30) + 1e-16) / 8.0]
    x = torch.stack(feats, -1).float().double()
    o = np.cumsum([nh * nin, nh, nh * nh, nh, nh])
    h = torch.relu(x @ w[:o[0]].view(nh, nin).T + w[o[0]:o[1]])
    h = torch.relu(h @ w[o[1]:o[2]].view(nh, nh).T + w[o[2]:o[3]])
    z = h @ w[o[3]:o[4]] + w[o[4]]
    raw = _pad_flags(z > math.log(thr / (1.0 - thr)), bc)
    ny, nx = raw.shape[0] - 4, raw.shape[1] - 4
    dil = torch.zeros((ny, nx), dtype=torch.bool, device=raw.device)
    for j in (1, 2, 3):
        for i in (1, 2, 3):
            dil |= raw[j:j + ny, i:i + nx]
    return _pad_flags(dil, bc)


def _xfaces(P, flag, T, eq, charwise, dt, dx, dy, corners):
    """x-face Gauss points (and corners) of a padded 2D state: lists over the points of (flux, state)."""
    ny, nx = P["W"].shape[1] - 4, P["W"].shape[2] - 4
    polys = []
    for a, b, s in (("W", "Y", 1.0), ("V", "Z", dx)):
        d = _stencil(T, P[a], dy * P[b], 0, ny + 2, 1)
        mix = _weights(T, _poly(T, d), d[0], d[1], d[2], flag if flag is True else flag[1:-1])
        polys.append([s * v for v in _combine(T, mix, d)])
    g = 0.5 * math.sqrt(0.6)
    W = P["W"]
    res = []
    for node in (-g, 0.0, g) + ((None,) if corners else ()):
        if node is None:
            E = [[0.5 * (a[:, :-1] + b[:, 1:]) for a, b in zip(_shift(p, 0.5), _shift(p, -0.5))] for p in polys]
            fl = flag if flag is True else flag[1:-2] | flag[2:-1]
        else:
            E = [[v[:, 1:-1] for v in _shift(p, node)] for p in polys]
            fl = flag if flag is True else flag[2:-2]
        basis = None
        if charwise:
            w = lambda r0, r1: 0.5 * (W[:, r0:r1, 1:-2] + W[:, r0:r1, 2:-1])
            ref = 0.5 * (w(1, -2) + w(2, -1)) if node is None else w(2, -2)
            _, R, L, _ = _eigen(list(ref))
            basis = (R, L)
        left, right = _sides(T, E[0], E[1], fl, basis, 2)
        res.append(_points(left, right, eq, dt, 1.0 / dx, 1.0 / dy))
    return res


def _turn(P, nc):
    """The state with x and y exchanged."""
    sw = lambda u: u.transpose(1, 2).contiguous() if nc == 1 else u.transpose(1, 2)[[0, 2, 1, 3]]
    return {"W": sw(P["W"]), "V": sw(P["Y"]), "Y": sw(P["V"]), "Z": sw(P["Z"])}


def _step(st, case, dom, bc, inflow, t, dt, T):
    """One step of size dt (W, V (, Y, Z) averages after it)."""
    eq, flow = _eq(case["flow"]), case["flow"]
    P = _pad(st, dom, bc, inflow, t, eq)
    nx = st["W"].shape[-1]
    dx = (dom[1] - dom[0]) / nx
    nc = st["W"].shape[0]
    flag = torch.zeros(P["W"].shape[1:], dtype=torch.bool, device=st["W"].device) if case["weights"] == "linear" else True
    if _dim(flow) == 1:
        basis = None
        if case["charwise"] and eq == S.EULER:
            _, R, L, _ = _eigen(list(0.5 * (P["W"][:, 1:-2] + P["W"][:, 2:-1])))
            basis = (R, L)
        left, right = _sides(T, [P["W"]], [dx * P["V"]], flag, basis, 1)
        F, We = _points(left, right, eq, dt, 1.0 / dx, None)
        return {"W": st["W"] - dt / dx * (F[:, 1:] - F[:, :-1]), "V": (We[:, 1:] - We[:, :-1]) / dx}
    ny = st["W"].shape[1]
    dy = (dom[3] - dom[2]) / ny
    if case["weights"] == "learned":
        flag = _learned_flags(P, dx, dy, bc)
    charwise = case["charwise"] and eq == S.EULER
    fx = _xfaces(P, flag, T, eq, charwise, dt, dx, dy, True)
    fy = _xfaces(_turn(P, nc), flag if flag is True else flag.T, T, eq, charwise, dt, dy, dx, False)
    wt = (5 / 18, 8 / 18, 5 / 18)
    FX, WX = (sum(w * r[k] for w, r in zip(wt, fx)) for k in (0, 1))
    back = (lambda u: u.transpose(1, 2)) if nc == 1 else (lambda u: u.transpose(1, 2)[[0, 2, 1, 3]])
    FY, WY = (back(sum(w * r[k] for w, r in zip(wt, fy))) for k in (0, 1))
    C = fx[3][1]
    return {"W": st["W"] - dt / dx * (FX[..., 1:] - FX[..., :-1]) - dt / dy * (FY[:, 1:] - FY[:, :-1]),
            "V": (WX[..., 1:] - WX[..., :-1]) / dx, "Y": (WY[:, 1:] - WY[:, :-1]) / dy,
            "Z": (C[:, 1:, 1:] - C[:, 1:, :-1] - C[:, :-1, 1:] + C[:, :-1, :-1]) / (dx * dy)}


def _march(case, flow, nx, ny, seed):
    """Steps of the reference from the seeded data: (state, time, steps)."""
    _, dom, bc, inflow = _flow(flow, seed)
    st, t, n = _initial(flow, nx, ny, seed), 0.0, 0
    case = {"weights": "plain", "charwise": False, "quintic": False, **case}
    T = _tables(case["quintic"])
    dx, dy = (dom[1] - dom[0]) / nx, (dom[3] - dom[2]) / ny
    end = case.get("t_final", math.inf)
    while t < end and n < case.get("steps", 10 ** 9):
        W = list(st["W"])
        if _eq(flow) == S.BURGERS:
            rate = W[0].abs() / dx + (W[0].abs() / dy if _dim(flow) == 2 else 0.0)
        else:
            _, u, v, _, c, _ = _prim(W)
            rate = (u.abs() + c) / dx + ((v.abs() + c) / dy if _dim(flow) == 2 else 0.0)
        dt = 0.6 / float(rate.max())
        if not dt <= end - t:
            dt = end - t
        st = _step(st, case, dom, bc, inflow, t, dt, T)
        t, n = t + dt, n + 1
    return st, t, n


def _train_exact(case, seed):
    x, y, params, m, v = (u.double() for u in _net_start(case, seed))
    nin, nh, pw, lr = S.FLAG_FEATURES, 32, 4.0, 2e-3
    p = params.clone().requires_grad_(True)
    o = np.cumsum([nh * nin, nh, nh * nh, nh, nh])
    h = torch.relu(x @ p[:o[0]].view(nh, nin).T + p[o[0]:o[1]])
    h = torch.relu(h @ p[o[1]:o[2]].view(nh, nh).T + p[o[2]:o[3]])
    z = h @ p[o[3]:o[4]] + p[o[4]]
    loss = (-pw * y * torch.nn.functional.logsigmoid(z) - (1 - y) * torch.nn.functional.logsigmoid(-z)).mean()
    loss.backward()
    g = p.grad
    m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    new = params - lr * (m / (1 - 0.9 ** 21)) / ((v / (1 - 0.999 ** 21)).sqrt() + 1e-8)
    return [loss.detach()[None], g, new, m, v]


def exact(case, seed):
    if case["kind"] == "train":
        return _train_exact(case, seed)
    if case["kind"] == "batch":  # the first problems: the whole ensemble would take minutes
        n = _sizes(case)
        return [None, [_march(case, case["flow"], k, k, 1000 * seed + i)[0] for i, k in enumerate(n[:FIRST])], None]
    st, t, n = _march(case, case["flow"], case["nx"], case["ny"], seed)
    return [st, t, n] if case["kind"] == "run" else [st]
