"""2D Euler over the gas constants, with cell data that jump from cell to cell: the fixed-point kernels hold gases of
gamma near 1.4 to 3 (csrc/ck_fixed.cuh) and leave the others to FP64; and over units of density and velocity far
below their exponents' range.  Against the oracle with the specification's tolerances
(tests/gpu_util.py), in all four readings of the reconstruction."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2304_09724_gb300 import shweno as S
from paper_2304_09724_gb300 import workloads as WL
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


def steep(gamma, nx, ny):
    rng = np.random.default_rng(77)
    rho, p = 10.0 ** rng.uniform(-0.2, 0.2, (2, ny, nx))
    # kinetic energies that stay below the internal one, p / (gamma - 1)
    u, v = rng.uniform(-0.3, 0.3, (2, ny, nx)) * np.sqrt(gamma) / max(1.0, gamma - 1.0)
    W = WL.euler_conserved(rho, u, p, v, gamma)
    return {"W": W, **{k: np.zeros_like(W) for k in "VYZ"}}


@pytest.mark.parametrize("gamma", [1.01, 1.1, 5.0 / 3.0, 3.0, 3.01, 7.0, 30.0, 1e3])
@pytest.mark.parametrize("opt", ["plain", "quintic", "charwise", "charwise quintic"])
def test_steep_cells(gamma, opt):
    nx, ny = 37, 22
    kw = dict(charwise="charwise" in opt, quintic="quintic" in opt)
    st = steep(gamma, nx, ny)
    dt = 4e-4 / np.sqrt(gamma)
    sol = S.Solver(2, S.EULER, nx, ny, gamma=gamma, **kw)
    sol.set_state(st)
    P = O.make_problem(2, S.EULER, nx, ny, 0.0, 1.0, 0.0, 1.0, gamma=gamma, **kw)
    o = st
    for _ in range(2):
        sol.step(dt)
        o = O.step(P, o, dt)
    g = sol.get_state()
    sol.close()
    wl = WL.vortex(8)
    wl.nx, wl.ny, wl.domain = nx, ny, (0.0, 1.0, 0.0, 1.0)
    U.check(g, o, "WVYZ", shocked=True, what=f"gamma {gamma:g} {opt}", wl=wl)


@pytest.mark.parametrize("er,ev", [(-330, 20), (-305, 0), (-290, -5), (30, -20), (20, 15)])
@pytest.mark.parametrize("opt", ["plain", "quintic", "charwise", "charwise quintic"])
@pytest.mark.parametrize("dim", [1, 2])
def test_units(er, ev, opt, dim):
    """Density 2^er and velocity 2^ev times that of an ordinary smooth flow."""
    kw = dict(charwise="charwise" in opt, quintic="quintic" in opt)
    nx, ny = 40, (1 if dim == 1 else 18)
    keys = "WV" if dim == 1 else "WVYZ"
    st = dict(zip(keys, WL.random_smooth_1d(5, nx) if dim == 1 else WL.random_smooth_2d(5, nx, ny)))
    power = [er] + [er + ev] * dim + [er + 2 * ev]
    f = np.ldexp(1.0, power).reshape((-1,) + (1,) * dim)
    st = {k: np.ascontiguousarray(v * f) for k, v in st.items()}
    dt = float(np.ldexp(0.003, -ev))
    args = (dim, S.EULER, nx, ny)
    sol = S.Solver(*args, **kw)
    sol.set_state(st)
    P = O.make_problem(*args, 0.0, 1.0, 0.0, 1.0, **kw)
    o = st
    for _ in range(2):
        sol.step(dt)
        o = O.step(P, o, dt)
    g = sol.get_state()
    sol.close()
    wl = WL.euler1d_sine(8) if dim == 1 else WL.vortex(8)
    wl.nx, wl.ny, wl.domain = nx, ny, (0.0, 1.0, 0.0, 1.0)
    U.check({k: v / f for k, v in g.items()}, {k: v / f for k, v in o.items()}, keys, shocked=False, what=f"2^{er} 2^{ev} {opt}", wl=wl)
