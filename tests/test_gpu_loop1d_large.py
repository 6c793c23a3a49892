"""The sliding 1D step loop (csrc/sv_loop1d.cu), which SV_LAUNCH_PERSISTENT takes on
grids beyond what the resident loop holds: bit for bit the per-step launches'
states, times and step counts, and an error status when a wait runs out."""
import math

import numpy as np
import pytest

from gpu_util import need_gpu
from paper_1805_03442_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    return need_gpu()


def beyond(prec, extra):
    """A size `extra` cells beyond the resident loop's: one block per SM (160 at most)
    of 20 warps of 60 cells, in double 8 warps of 28."""
    import torch
    sms = min(torch.cuda.get_device_properties(0).multi_processor_count, 160)
    return sms * (8 * 28 if prec == "FP64" else 20 * 60) + extra


def both(sv, P, N, U0, nsteps=None, t_end=None, bc=(0, 0), drive=None):
    out = []
    for mode in (sv.LAUNCH_PER_STEP, sv.LAUNCH_PERSISTENT):
        with sv.Solver(P, (N,), (1.0,), bc=bc) as s:
            s.set_launch(mode)
            assert s.launch == mode
            if drive is not None:
                s.set_drive(*drive)
            s.write_state(U0)
            rc = 0
            if t_end is None:
                s.step(nsteps)
            else:
                rc, _ = s.run_to(t_end, check=False)
            U, t = s.read_state()
            out.append((U, t, s.time()[1], s.status(), rc))
    (U, *a), (V, *b) = out
    assert a == b and np.array_equal(U, V, equal_nan=True)
    return out[1]


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("limiter", ["MINMOD", "VANLEER", "MC"])
@pytest.mark.parametrize("src", ["frozen", "qi_zero", "general"])
def test_limiters_and_sources(sv, prec, limiter, src):
    over = {"frozen": dict(tau0=math.inf), "qi_zero": dict(),
            "general": dict(Q_rho=0.5, Q_T=-0.7, I_rho=1.0, I_T=0.6)}[src]
    N = beyond(prec, 1)
    P = sv.Params(precision=getattr(sv, prec), limiter=getattr(sv, limiter), **over)
    both(sv, P, N, inputs.random_states(1, N, seed=7, smooth=True), nsteps=4)


@pytest.mark.parametrize("prec, bc", [("FP64", (1, 1)), ("FP32", (2, 2)), ("FP32_PC", (1, 2)), ("FP64", (2, 1))])
def test_walls_outflow(sv, prec, bc):
    N = beyond(prec, 63)
    P = sv.Params(precision=getattr(sv, prec), tau0=0.3)
    both(sv, P, N, inputs.random_states(1, N, seed=11, smooth=True), nsteps=5, bc=bc)


@pytest.mark.parametrize("prec", ["FP32_PS", "FP64"])
def test_driven(sv, prec):
    N = beyond(prec, 100)
    P = sv.Params(precision=getattr(sv, prec))
    ev0 = P.Ck + P.S
    U0 = inputs.waves_1d(1.4, N, 1.0, inputs.equilibrium_primitive(0.1, 1.0), [])
    base = [1.0, 0.0, 1.0 / 0.4 + ev0, ev0]
    amp = [1e-3, 1e-3, 1e-3 / 0.4 * 1.4, 1e-4]
    both(sv, P, N, U0, nsteps=7, bc=(3, 2), drive=(20.0, 17.0 - 0.3j, base, amp))


def test_stops_at_t_end_and_at_a_nonphysical_state(sv):
    N = beyond("FP64", 5)
    P = sv.Params(precision=sv.FP64, tau0=0.2)
    r = both(sv, P, N, inputs.random_states(1, N, seed=3, smooth=True), t_end=8.4 / N)
    assert r[1] == 8.4 / N and r[4] == 0 and r[2] > 3
    # two streams flying apart, the medium's times scaled with the cell: a near-vacuum
    # that goes non-physical after a few dozen steps
    P = sv.Params(precision=sv.FP64, tau0=100.0 / N)
    x = inputs.cell_centres(N, 1.0)
    v = np.where(x < 0.5, -3.0, 3.0)
    U0 = inputs.prim_to_cons(1.4, np.ones(N), [v], np.full(N, 1e-2), np.full(N, 0.5))
    r = both(sv, P, N, U0, t_end=25.0 / N)
    assert r[4] in (sv.SV_ENONPHYS, sv.SV_EDT) and r[3] != 0


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
def test_barrier_wait_limit_ends_with_estall(sv, prec):
    """With the wait limited to one poll the blocks that arrive before the last one
    give up, raise the stall flag and leave; the launch ends with SV_ESTALL.  After
    an upload and with the default limit the solver steps as a per-step one."""
    N = beyond(prec, 640)
    P = sv.Params(precision=getattr(sv, prec))
    U0 = inputs.random_states(1, N, seed=5, smooth=True)
    with sv.Solver(P, (N,), (1.0,)) as s:
        s.set_launch(sv.LAUNCH_PERSISTENT)
        s.write_state(U0)
        s.set_wait_limit(1)
        rc, _ = s.run_to(20.0 / N, check=False)
        assert rc == sv.SV_ESTALL and s.status() & sv.FLAG_STALL
        s.set_wait_limit(0)
        s.write_state(U0)
        assert s.status() == 0
        rc, k = s.run_to(20.0 / N, check=False)
        U, t = s.read_state()
        assert rc == 0 and s.status() == 0
    with sv.Solver(P, (N,), (1.0,)) as r:
        r.set_launch(sv.LAUNCH_PER_STEP)
        r.write_state(U0)
        rc, k2 = r.run_to(20.0 / N, check=False)
        V, t2 = r.read_state()
    assert rc == 0 and (k, t) == (k2, t2) and np.array_equal(U, V)
