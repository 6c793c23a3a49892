"""The resident 1D step loop when a wait for another block runs out
(sv_set_wait_limit): the launch ends, the stall flag says so, and nothing that
is reported as good differs from per-step launches."""
import numpy as np
import pytest

from gpu_util import need_gpu
from paper_1805_03442_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    return need_gpu()


def per_step(sv, P, N, U0, k):
    with sv.Solver(P, (N,), (1.0,)) as r:
        r.set_launch(sv.LAUNCH_PER_STEP)
        r.write_state(U0)
        r.step(k)
        return r.read_state()


@pytest.mark.parametrize("prec, N", [("FP32", 182400), ("FP32", 4000), ("FP64", 34048)])
def test_blocks_that_start_late(sv, prec, N):
    """Blocks that start while others have given up already: every thread of a
    block leaves or stays with it.  Each launch ends, and the solver steps as a
    fresh one after an upload."""
    P = sv.Params(precision=getattr(sv, prec), tau0=0.3)
    U0 = inputs.random_states(1, N, seed=N, smooth=True)
    want, t = per_step(sv, P, N, U0, 4)
    with sv.Solver(P, (N,), (1.0,)) as s:
        s.set_launch(sv.LAUNCH_PERSISTENT)
        s.set_wait_limit(1)
        stalled = 0
        for _ in range(40):
            s.write_state(U0)
            s.step(50)
            stalled += bool(s.status() & sv.FLAG_STALL)
        assert stalled
        s.set_wait_limit(0)
        s.write_state(U0)
        s.step(4)
        U, tu = s.read_state()
        assert s.status() == 0 and tu == t and np.array_equal(U, want)


@pytest.mark.parametrize("prec, N, k", [("FP32", 4000, 2), ("FP32", 4000, 3), ("FP64", 1600, 1), ("FP64", 1600, 2)])
def test_stall_of_the_last_step_is_kept(sv, prec, N, k):
    """Runs of few steps with waits of few polls: a block that gives up in the last
    step leaves its cells unwritten while the others finish.  The stall flag
    stays, or the state, time and step count are those of per-step launches."""
    P = sv.Params(precision=getattr(sv, prec), tau0=0.3)
    U0 = inputs.random_states(1, N, seed=N, smooth=True)
    want, t = per_step(sv, P, N, U0, k)
    seen = set()
    with sv.Solver(P, (N,), (1.0,)) as s:
        s.set_launch(sv.LAUNCH_PERSISTENT)
        for polls in (1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 64, 256, 4096):
            s.set_wait_limit(polls)
            for _ in range(30):
                s.write_state(U0)
                s.step(k)
                U, tu = s.read_state()
                bad = s.status()
                seen.add(bad)
                if not bad & sv.FLAG_STALL:
                    assert bad == 0 and tu == t and s.time()[1] == k
                    assert np.array_equal(U, want), (polls, int((U != want).any(axis=0).sum()))
    assert sv.FLAG_STALL in seen and 0 in seen
