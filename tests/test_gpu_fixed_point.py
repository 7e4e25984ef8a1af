"""The Cauchy-Kovalevskaya procedure in block fixed point (csrc/fixed.cuh, ck_fixed.cuh), where it
can go wrong: points per CTA around the 16-, 64- and 127-point edges of its warps, meshes whose
widths differ, units far from 1, extreme gas constants, steep data (coefficients that grow with
the degree and repeat the recursion in another scale), a uniform state.  Against the oracle with the
specification's tolerances (tests/gpu_util.py): the fixed-point form rounds finer than FP64."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2304_09724_gb300 import shweno as S
from paper_2304_09724_gb300 import workloads as WL
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


def both(state, nx, ny, dt, steps, eq=S.EULER, domain=(0.0, 1.0, 0.0, 1.0), bc=(0, 0, 0, 0), gamma=1.4):
    sol = S.Solver(2, eq, nx, ny, domain, bc, gamma=gamma)
    sol.set_state(state)
    P = O.make_problem(2, eq, nx, ny, *domain, gamma=gamma, bc=bc)
    o = state
    for _ in range(steps):
        sol.step(dt)
        o = O.step(P, o, dt)
    g = sol.get_state()
    sol.close()
    return g, o


def smooth(nx, ny, eq=S.EULER, seed=11):
    return {k: v.copy() for k, v in zip("WVYZ", WL.random_smooth_2d(seed, nx, ny, eq=eq))}


def compare(g, o, nx, ny, domain=(0.0, 1.0, 0.0, 1.0), shocked=False, what=""):
    wl = WL.vortex(8)
    wl.nx, wl.ny, wl.domain = nx, ny, domain
    U.check(g, o, "WVYZ", shocked=shocked, what=what, wl=wl)


@pytest.mark.parametrize("n", [14, 15, 16, 31, 62, 63, 64, 79, 126, 127, 128])
@pytest.mark.parametrize("eq", [S.EULER, S.BURGERS])
def test_points_per_cta(n, eq):
    for nx, ny in ((n, 5), (5, n)):
        st = smooth(nx, ny, eq)
        g, o = both(st, nx, ny, 0.1 / n, 2, eq)
        compare(g, o, nx, ny, what=f"{nx}x{ny}")


@pytest.mark.parametrize("domain", [(0.0, 3.0, 0.0, 1.0), (0.0, 1.0, 0.0, 7.0)])
def test_unequal_widths(domain):
    st = smooth(24, 20)
    st["V"] /= domain[1]
    st["Y"] /= domain[3]
    st["Z"] /= domain[1] * domain[3]
    g, o = both(st, 24, 20, 0.004, 2, domain=domain)
    compare(g, o, 24, 20, domain, what=str(domain))


@pytest.mark.parametrize("rho,vel", [(1e-40, 1e30), (1e12, 1e-14), (1.0, 1e6), (1e-3, 1e-9)])
def test_units(rho, vel):
    st = smooth(22, 18)
    f = np.array([rho, rho * vel, rho * vel, rho * vel * vel])[:, None, None]
    g, o = both({k: v * f for k, v in st.items()}, 22, 18, 0.004 / vel, 2)
    compare({k: v / f for k, v in g.items()}, {k: v / f for k, v in o.items()}, 22, 18, what=f"rho {rho} vel {vel}")


@pytest.mark.parametrize("gamma", [1.02, 3.0, 6.5, 20.0])
def test_gas_constant(gamma):
    st = smooth(20, 16)
    kin = 0.5 * (st["W"][1] ** 2 + st["W"][2] ** 2) / st["W"][0]
    st["W"][3] = kin + (st["W"][3] - kin) * 0.4 / (gamma - 1.0)
    for k in "VYZ":
        st[k][3] *= 0.4 / (gamma - 1.0)
    g, o = both(st, 20, 16, 0.003, 2, gamma=gamma)
    compare(g, o, 20, 16, what=f"gamma {gamma}")


@pytest.mark.parametrize("seed", range(4))
@pytest.mark.parametrize("eq", [S.EULER, S.BURGERS])
def test_steep_cells(seed, eq):
    """Cell data that jump from cell to cell by up to a factor of 6 (no smooth scale at all)."""
    rng = np.random.default_rng(900 + seed)
    nx, ny = 41, 23
    if eq == S.BURGERS:
        W = rng.uniform(-1.0, 1.0, (1, ny, nx)) * 10.0 ** rng.uniform(-6, 0, (1, ny, nx))
    else:
        rho, p = 10.0 ** rng.uniform(-0.4, 0.4, (2, ny, nx))
        u, v = rng.uniform(-0.3, 0.3, (2, ny, nx))
        W = WL.euler_conserved(rho, u, p, v)
    st = {"W": W, "V": np.zeros_like(W), "Y": np.zeros_like(W), "Z": np.zeros_like(W)}
    g, o = both(st, nx, ny, 2e-4, 2, eq, bc=(WL.OUTFLOW, WL.REFLECTIVE, WL.OUTFLOW, WL.OUTFLOW))
    compare(g, o, nx, ny, shocked=True, what=f"steep {seed}")


def test_uniform_state_stays():
    nx, ny = 20, 12
    c = WL.constant_state(2, S.EULER, nx, ny)
    g, _ = both(c, nx, ny, 0.004, 2)
    assert np.array_equal(g["W"], c["W"]) and all(np.all(g[k] == 0.0) for k in "VYZ")
