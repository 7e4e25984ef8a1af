"""What a batch keeps between runs and shares with its handles: the CFL number of its cached graph is its own,
whatever other batches ran in between."""
import pytest

from paper_2304_09724_gb300 import shweno as S
from paper_2304_09724_gb300 import workloads as WL
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


def steps_of(batch, sol, wl, cfl):
    sol.set_state(wl.state)
    n = sol.time()[1]
    batch.run(0.05, cfl)
    return sol.time()[1] - n


def test_each_batch_keeps_its_own_cfl():
    wl = WL.euler1d_sine(200)
    a, b, solo = (U.solver_of(wl) for _ in range(3))
    A, B = S.Batch([a]), S.Batch([b])
    want = {}
    for cfl in (0.6, 0.3):
        solo.set_state(wl.state)
        want[cfl] = solo.run(0.05, cfl)[1]
    assert want[0.3] > 1.5 * want[0.6]
    got = [steps_of(batch, sol, wl, cfl) for batch, sol, cfl in ((A, a, 0.6), (B, b, 0.3), (A, a, 0.3), (B, b, 0.6), (A, a, 0.3))]
    assert got == [want[c] for c in (0.6, 0.3, 0.3, 0.6, 0.3)]
    for x in (A, B, a, b, solo):
        x.close()
