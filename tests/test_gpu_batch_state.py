"""What a batch keeps between runs and shares with its handles: the CFL number of its cached graph is its own,
whatever other batches ran in between; a run starts after what is in flight on the handles' streams."""
import numpy as np
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


@pytest.mark.parametrize("mode", [S.BATCH_PERSISTENT, S.BATCH_LOCKSTEP])
@pytest.mark.parametrize("tune", [False, True])
def test_run_starts_after_the_handles_streams(mode, tune):
    """States set on streams that are still busy (a tenth of a second) when the batch runs, twice in a row."""
    import torch
    wls = [WL.euler1d_sine(4000), WL.vortex(48), WL.euler1d_sine(900)]
    streams = [torch.cuda.Stream() for _ in wls]
    sols = [U.solver_of(wl, stream=st.cuda_stream) for wl, st in zip(wls, streams)]
    want = []
    for wl in wls:
        s = U.solver_of(wl)
        s.set_state(wl.state)
        S.shweno_advance(s.h, 3, wl.cfl)
        want.append((s.get_state(), s.time()))
        s.close()
    b = S.Batch(sols)
    b.set_mode(mode)
    dev = [{k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in wl.state.items()} for wl in wls]
    torch.cuda.synchronize()
    for _ in range(2):
        for sol, st, d in zip(sols, streams, dev):
            with torch.cuda.stream(st):
                torch.cuda._sleep(200_000_000)
            sol.set_state(d)
        if tune:
            b.autotune(1e9, wls[0].cfl, trial_steps=1)
        b.run(1e9, wls[0].cfl, max_steps=3)
        for sol, wl, (o, time) in zip(sols, wls, want):
            assert sol.time()[1] == time[1] and abs(sol.time()[0] - time[0]) <= 1e-12 * time[0]
            U.check(sol.get_state(), o, U.fields(wl), shocked=False, what=wl.name, wl=wl)
    b.close()
    for s in sols:
        s.close()
