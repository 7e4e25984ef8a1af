"""Cells whose neighbours are larger by many orders of magnitude.  The second pass of 2D Euler holds a
cell's data in one scale per component; where that would cost the smaller cells bits that FP64 has, the
pass runs in FP64 (cell_exponents, face_setup_fx of csrc/step2d_items.cuh).  A block of hot, dense or fast
gas in a quiet smooth flow, one short step, the quiet cells by themselves: every cell and component
against the oracle, by the size that the component has in the quiet part.  Tolerances: the
specification's (tests/gpu_util.py), relative to the quiet part."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2304_09724_gb300 import shweno as S
from paper_2304_09724_gb300 import workloads as WL
from tests import gpu_util as U

pytestmark = pytest.mark.gpu

NX, NY = 150, 24  # x-faces of a row: one CTA of 127 and one of rows' remainders; the block is in some of them
BLOCK = np.s_[9:15, 40:49]


def blocked(kind, ratio):
    """Quiet smooth flow with a block of uniform gas of `ratio` times its energy, density, or velocity
    (at the same Mach number)."""
    st = {k: v.copy() for k, v in zip("WVYZ", WL.random_smooth_2d(3, NX, NY))}
    rho, p, u, v = {"energy": (1.0, ratio, 0.4, -0.3), "density": (ratio, 1.0, 0.4, -0.3),
                    "speed": (1.0, ratio * ratio, ratio, 0.5 * ratio)}[kind]
    b = WL.euler_conserved(*(np.full((6, 9), x) for x in (rho, u, p, v)))
    st["W"][(slice(None), *BLOCK)] = b
    for k in "VYZ":
        st[k][(slice(None), *BLOCK)] = 0.0
    hot = np.zeros((NY, NX), bool)
    hot[BLOCK] = True
    near = np.zeros_like(hot)  # the block and the cells with a face on it
    for dj in (-1, 0, 1):
        for di in (-1, 0, 1):
            near |= np.roll(hot, (dj, di), (0, 1))
    speed = max(u, 1.0) + (1.4 * p / rho) ** 0.5
    return st, ~near, 1e-3 / (NX * speed), near


def check_quiet(g, o, quiet, what):
    dx, dy = 1.0 / NX, 1.0 / NY
    for q in range(4):
        wmax = np.max(np.abs(o["W"][q][quiet]))
        for k in "WVYZ":
            d, ref = np.abs(g[k][q] - o[k][q])[quiet], np.max(np.abs(o[k][q][quiet]))
            tol = U.SMOOTH_TOL * ref + U.deriv_floor(k, wmax, dx, dy)
            if k == "W":
                tol = 1e-13 * ref  # a short step: the sum of one state and a small change
            assert np.max(d) <= tol, f"{what} {k}[{q}]: {np.max(d) / tol:.1f} times the tolerance"


@pytest.mark.parametrize("kind,ratio", [(k, r) for k in ("energy", "density") for r in (30.0, 1e4, 1e6, 1e9, 1e12)]
                         + [("speed", 30.0)])
@pytest.mark.parametrize("flags", [False, True])
def test_quiet_side_of_a_jump(kind, ratio, flags):
    st, quiet, dt, near = blocked(kind, ratio)
    flag = None
    if flags:  # nonlinear weights at the block, either kind elsewhere
        flag = (np.random.default_rng(5).random((NY, NX)) < 0.5).astype(np.uint8)
        for dj in (-1, 0, 1):
            for di in (-1, 0, 1):
                flag |= np.roll(near, (dj, di), (0, 1)).astype(np.uint8)
    sol = S.Solver(2, S.EULER, NX, NY, flag_mode=2 if flags else 0)
    sol.set_state(st)
    if flags:
        sol.set_flags(flag)
    sol.step(dt)
    g = sol.get_state()
    sol.close()
    o = O.step(O.make_problem(2, S.EULER, NX, NY, 0.0, 1.0, 0.0, 1.0), st, dt, flag=flag)
    check_quiet(g, o, quiet, f"{kind} {ratio:g}")


@pytest.mark.parametrize("mode", [S.BATCH_PERSISTENT, S.BATCH_LOCKSTEP])
def test_quiet_side_in_a_batch(mode):
    sols, refs = [], []
    for kind, ratio in (("energy", 1e9), ("density", 1e6)):
        st, quiet, dt, _ = blocked(kind, ratio)
        sol = S.Solver(2, S.EULER, NX, NY)
        sol.set_state(st)
        P = O.make_problem(2, S.EULER, NX, NY, 0.0, 1.0, 0.0, 1.0)
        refs.append((O.step(P, st, dt), quiet, dt))
        sols.append(sol)
    b = S.Batch(sols)
    b.set_mode(mode)
    # one step to the end time: the CFL number never limits it
    b.run([dt for _, _, dt in refs], 1e3, max_steps=1)
    for sol, (o, quiet, dt) in zip(sols, refs):
        assert sol.time() == (dt, 1)
        check_quiet(sol.get_state(), o, quiet, f"batch mode {mode}")
    b.close()
    for sol in sols:
        sol.close()


@pytest.mark.parametrize("gam", [(0.1, 0.45, 0.45), (0.2, 0.5, 0.3), (0.26, 0.37, 0.37), (0.6, 0.2, 0.2)])
def test_linear_weights_of_any_size(gam):
    """A cell's p1 carries up to 1 / gam[0]: 10 and 5 are out of the fixed-point format, 3.8 and 1.7 in it."""
    st, _, dt, _ = blocked("energy", 3.0)
    h = S.shweno_create(S.make_grid(2, S.EULER, NX, NY), 1.4, S.make_bc((0, 0, 0, 0)), S.make_opts(gam=gam))
    S.shweno_set_state(h, *(np.ascontiguousarray(st[k]) for k in "WVYZ"))
    P = O.make_problem(2, S.EULER, NX, NY, 0.0, 1.0, 0.0, 1.0, gam=gam)
    o = st
    for _ in range(2):
        S.shweno_step(h, 300.0 * dt)
        o = O.step(P, o, 300.0 * dt)
    g = {k: np.empty_like(st[k]) for k in "WVYZ"}
    S.shweno_get_state(h, *(g[k] for k in "WVYZ"))
    S.shweno_destroy(h)
    wl = WL.vortex(8)
    wl.nx, wl.ny, wl.domain = NX, NY, (0.0, 1.0, 0.0, 1.0)
    U.check(g, o, "WVYZ", shocked=True, what=f"gam {gam}", wl=wl)
