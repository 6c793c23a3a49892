"""Non-finite states in double are flagged, whichever kernel bounds them: an
infinite pressure or a NaN of either sign in an uploaded state, and the NaN that a
step makes of a half-step state without pressure (the closures of eq. 6 at T < 0)."""
import types

import numpy as np
import pytest

from gpu_util import need_gpu, oracle_params
from oracle import orc as O
from paper_1805_03442_gb300 import inputs

pytestmark = pytest.mark.gpu

GRIDS = [(101,), (20000,), (100000,), (64, 40), (20, 16, 12)]
OVER = [dict(tau0=0.3), dict(tau0=0.3, tau_T=-1.3), dict(tau0=float("inf"), S=0.0)]
# heating that takes a half step's E_nu past its E, with no cap on dt by tau
HEATED = dict(tau0=0.01, c_tau=1e9)


@pytest.fixture(scope="module")
def sv():
    return need_gpu()


def states(dim, ncell, field, value):
    U = inputs.random_states(dim, ncell, seed=3, smooth=True)
    U[field, ncell // 2] = value
    return U


def bad_flags(sv):
    return sv.FLAG_DT | sv.FLAG_NONPHYS


@pytest.mark.parametrize("over", OVER)
@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("what", ["E inf", "E_nu -inf", "rho nan", "v nan", "E nan", "E_nu nan", "E -nan"])
def test_upload_and_step(sv, n, over, what):
    dim, ncell = len(n), int(np.prod(n))
    name, value = what.split()
    field = {"rho": 0, "v": 1, "E": dim + 1, "E_nu": dim + 2}[name]
    # both signs of the NaN: a NaN's own is not kept by every conversion from text
    v = np.copysign(np.nan, -1.0 if value == "-nan" else 1.0) if "nan" in value else float(value)
    P = sv.Params(precision=sv.FP64, **over)
    with sv.Solver(P, n, tuple(m / n[0] for m in n)) as s:
        s.write_state(states(dim, ncell, field, v))
        assert s.status() & bad_flags(sv)
        s.step(2)
        assert s.time()[1] == 0


def heated(sv, n, method=None):
    """A state at rest with little vibrational energy and a pump S that takes E_nu
    past E = 2.5 + 0.1 within half a step of dt = 0.4 h / c."""
    h = 1.0 / n[0]
    S = 40.0 * 0.01 / (0.2 * h / np.sqrt(1.4))
    over = dict(HEATED, S=S)
    P = sv.Params(precision=sv.FP64, **over)
    one = np.ones(int(np.prod(n)))
    U = inputs.prim_to_cons(1.4, one, [0 * one] * len(n), one, 0.1 * one)
    return P, U


@pytest.mark.parametrize("n", GRIDS)
def test_half_step_without_pressure(sv, n):
    P, U = heated(sv, n)
    with sv.Solver(P, n, tuple(m / n[0] for m in n)) as s:
        s.write_state(U)
        assert s.status() == 0
        s.step(1)
        assert s.status() & sv.FLAG_NONPHYS and s.time()[1] == 1
        s.step(3)
        assert s.time()[1] == 1
        assert s.run_to(1.0, check=False)[0] == sv.SV_ENONPHYS
    if len(n) == 1:
        with sv.Solver(P, n, (1.0,)) as s:
            s.set_launch(sv.LAUNCH_PER_STEP)
            s.write_state(U)
            s.step(3)
            assert s.status() & sv.FLAG_NONPHYS and s.time()[1] == 1
    h = 1.0 / n[0]
    if len(n) == 1 and n[0] < 1000:
        Po = oracle_params(P)
        assert O.step(Po, U, n[0], h, O.dt_cfl(Po, U, n[0], h))[1] != 0


@pytest.mark.parametrize("n", [1000, 5000])
def test_allocation_free_step(sv, n):
    torch = pytest.importorskip("torch")
    U = torch.from_numpy(states(1, n, 2, np.inf)).cuda()
    out = torch.empty_like(U)
    _, flags = sv.step1d_noalloc(sv.Params(precision=sv.FP64, tau0=0.3), n, 1.0, U.data_ptr(), out.data_ptr())
    assert flags & bad_flags(sv)
    P, U0 = heated(sv, (n,))
    U = torch.from_numpy(U0).cuda()
    _, flags = sv.step1d_noalloc(P, n, 1.0, U.data_ptr(), out.data_ptr())
    assert flags & sv.FLAG_NONPHYS


def test_batch(sv):
    """Runs that stop at once (an infinity), at the first step (a half step without
    pressure) and at their end, on windows in registers and streamed."""
    P, _ = heated(sv, (300,))
    kinds = [("inf", 300), ("inf", 20000), ("heated", 300), ("heated", 20000), ("good", 400)]
    runs, U = [], []
    for kind, n in kinds:
        S, tau0 = (1.0, 0.3) if kind != "heated" else (heated(sv, (n,))[0].S, 0.01)
        runs.append(types.SimpleNamespace(n=n, L=1.0, S=S, tau0=tau0, tau_rho=-1.0, tau_T=-1.5, Q_rho=0.0,
                                          Q_T=0.0, I_rho=0.0, I_T=0.0, t_end=0.01, m=1))
        U.append(heated(sv, (n,))[1] if kind == "heated" else
                 states(1, n, 2, np.inf) if kind == "inf" else
                 inputs.waves_1d(1.4, n, 1.0, inputs.equilibrium_primitive(0.1, 1.0), []))
    with sv.Batch(P, runs, U, log_cap=4) as b:
        b.run()
        b.sync()
        got = [b.read(i)[2:] for i in range(len(kinds))]
    for (kind, _), (steps, flags) in zip(kinds, got):
        if kind == "good":
            assert flags == 0 and steps > 1
        else:
            assert flags & bad_flags(sv) and steps == (1 if kind == "heated" else 0)
