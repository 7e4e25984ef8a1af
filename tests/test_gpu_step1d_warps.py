"""The 1D step kernel at the edges of its warps (30 cells each) and of its launch rules: one cell
more or less than a warp, than two, than one CTA of four warps per SM (152 warps, 4560 cells), than
two of them (304 warps, 9120 cells: the Euler kernel changes there) and than 1216 warps (36480 cells: four warps per CTA from there on); both
equations, both readings of p1, both kinds of ends.  Against the oracle with the specification's
tolerances (tests/gpu_util.py)."""
import pytest

from paper_2304_09724_gb300 import workloads as WL
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [4, 29, 30, 31, 59, 60, 61, 119, 121, 4559, 4560, 4561, 9120, 9121, 36480, 36481])
@pytest.mark.parametrize("eq", [WL.BURGERS, WL.EULER])
def test_warp_and_launch_edges(n, eq):
    W, V = WL.random_smooth_1d(n, n, eq=eq)
    for quintic in (False, True) if n < 5000 else (n % 2 == 1,):
        wl = WL.burgers_sine(n) if eq == WL.BURGERS else WL.euler1d_sine(n)
        wl.domain = (0.0, 1.0, 0.0, 1.0)
        if n % 2:
            wl.bc = (WL.OUTFLOW, WL.OUTFLOW, 0, 0)
        wl.state = {"W": W, "V": V}
        g, o = U.steps_both(wl, [0.1 / n] * 2, quintic=quintic)
        U.check(g, o, U.fields(wl), shocked=False, what=f"eq={eq} n={n} quintic={quintic}", wl=wl)
