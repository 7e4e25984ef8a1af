"""A slow shear flow: fast smooth flow in one direction, nothing varies in the other, along which the gas drifts
at 2^-10 to 2^-40 of the sound speed.  The pressure does not act on the drift, so FP64 carries it with all
its bits; the library's fixed-point kernels have to as well (csrc/step2d_items.cuh: cell_exponents and
ck_coarse2d send such points to FP64).  The drift by itself, with the specification's tolerances
(tests/gpu_util.py) relative to the drift: down to 2^-20 against the oracle; below, where the oracle's own noise
(2e-19 of the sound speed with contracted multiply-adds) would show in the slopes, against the same
flow at 2^-20, with which it scales."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2304_09724_gb300 import shweno as S
from paper_2304_09724_gb300 import workloads as WL
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


def shear(n, m, drift, axis):
    """n cells along the flow (x for axis 0, y for 1), m across; the drift is along the other axis."""
    def f(x, y):
        s = (x, y)[axis] + 0.0 * (x + y)
        w = lambda k, ph: np.sin(2 * np.pi * k * s + ph)
        fast, slow = 0.5 + 0.1 * w(1, 0.3), drift * (1.0 + 0.3 * w(2, 1.1))
        u, v = (fast, slow) if axis == 0 else (slow, fast)
        return WL.euler_conserved(1.0 + 0.1 * w(1, 0.0), u, 1.0 + 0.1 * w(1, 2.0), v)
    nx, ny = (n, m) if axis == 0 else (m, n)
    st = {}
    for k, v in zip("WVYZ", WL.project_2d(f, 0.0, 1.0, 0.0, 1.0, nx, ny)):
        even = k == "W" or k == "VY"[axis]  # the same bits in every cell across the flow, no slope there
        st[k] = np.repeat(v.take([0], axis=1 + axis), m, axis=1 + axis) if even else np.zeros((4, ny, nx))
    return st, nx, ny


@pytest.mark.parametrize("bits", [10, 20, 26, 30, 40])
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("opt", ["plain", "quintic", "charwise", "charwise quintic"])
def test_drift_keeps_its_bits(bits, axis, opt):
    kw = dict(charwise="charwise" in opt, quintic="quintic" in opt)
    ref = min(bits, 20)

    def library(bits):
        st, nx, ny = shear(40, 6, 2.0 ** -bits, axis)
        sol = S.Solver(2, S.EULER, nx, ny, **kw)
        sol.set_state(st)
        for _ in range(3):
            sol.step(0.004)
        g = sol.get_state()
        sol.close()
        return g, nx, ny

    g, nx, ny = library(bits)
    if bits > ref:
        o = library(ref)[0]
    else:
        o = shear(40, 6, 2.0 ** -bits, axis)[0]
        P = O.make_problem(2, S.EULER, nx, ny, 0.0, 1.0, 0.0, 1.0, **kw)
        for _ in range(3):
            o = O.step(P, o, 0.004)
    wl = WL.vortex(8)
    wl.nx, wl.ny, wl.domain = nx, ny, (0.0, 1.0, 0.0, 1.0)
    q, along = 2 - axis, "WV" if axis == 0 else "WY"
    scale = 2.0 ** (bits - ref)
    U.check({k: g[k][q] * scale for k in along}, {k: o[k][q] for k in along}, along, shocked=False, what=f"drift 2^-{bits}", wl=wl)
    rest = [p for p in range(4) if p != q]
    U.check({k: g[k][rest] for k in "WVYZ"}, {k: o[k][rest] for k in "WVYZ"}, "WVYZ", shocked=False, what=f"flow at drift 2^-{bits}", wl=wl)
