"""The resident 1D step loop (csrc/sv_res1d.cuh) against per-step launches, bit
for bit, at the edges of its decomposition: one warp or block more or less, odd
sizes, the smallest grids of every boundary, its capacity, and launches that
follow one another."""
import numpy as np
import pytest

from gpu_util import need_gpu
from paper_1805_03442_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    return need_gpu()


def pair(sv, P, N, U0, go, bc=(0, 0), drive=None, modes=None):
    out = []
    for mode in (sv.LAUNCH_PER_STEP,) + (modes or (sv.LAUNCH_AUTO, sv.LAUNCH_PERSISTENT)):
        with sv.Solver(P, (N,), (1.0,), bc=bc) as s:
            s.set_launch(mode)
            if drive is not None:
                s.set_drive(*drive)
            s.write_state(U0)
            extra = go(s)
            U, t = s.read_state()
            out.append((U, t, s.time()[1], s.status(), s.dt(), extra))
    for o in out[1:]:
        assert np.array_equal(o[0], out[0][0], equal_nan=True)
        assert o[1:] == out[0][1:]
    return out[0]


# 60 cells per warp in float, 28 in double; 12 / 4 warps in a lone block, 4 / 3
# in the others; capacities 152 * 20 * 60 and 152 * 8 * 28 on a GB300
@pytest.mark.parametrize("N", [2, 3, 4, 59, 60, 61, 121, 719, 721, 961, 14401, 182399, 182400, 182401])
@pytest.mark.parametrize("prec", ["FP32", "FP32_PS"])
def test_float_sizes(sv, N, prec):
    P = sv.Params(precision=getattr(sv, prec), tau0=0.3)
    pair(sv, P, N, inputs.random_states(1, N, seed=N, smooth=True), lambda s: s.step(9))


@pytest.mark.parametrize("N", [2, 3, 27, 28, 29, 111, 113, 169, 34047, 34048, 34049])
def test_double_sizes(sv, N):
    P = sv.Params(precision=sv.FP64, tau0=0.3)
    pair(sv, P, N, inputs.random_states(1, N, seed=N, smooth=True), lambda s: s.step(7))


@pytest.mark.parametrize("bc", [(1, 1), (2, 2), (1, 2), (2, 1), (0, 2), (3, 1)])
@pytest.mark.parametrize("N", [2, 3, 61, 1000])
@pytest.mark.parametrize("prec", ["FP32_PC", "FP64"])
def test_boundaries(sv, bc, N, prec):
    P = sv.Params(precision=getattr(sv, prec), tau0=0.3)
    ev0 = P.Ck + P.S
    drive = (20.0, 17.0 - 0.3j, [1.0, 0.0, 2.5 + ev0, ev0], [1e-3, 1e-3, 3.5e-3, 1e-4])
    pair(sv, P, N, inputs.random_states(1, N, seed=N, smooth=True), lambda s: s.step(8), bc=bc,
         drive=drive if bc[0] == 3 else None)


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("N", [500, 5000])
def test_launches_in_a_row(sv, prec, N):
    """Runs of a few steps, clamped end times and single steps between them:
    the exchange words of one launch are never taken for the next one's."""
    P = sv.Params(precision=getattr(sv, prec), limiter=sv.VANLEER)
    modes = inputs.random_phase_modes(2, inputs.acoustic_shape(1.4), 4, 1, 1e-2)
    U0 = inputs.waves_1d(1.4, N, 1.0, inputs.equilibrium_primitive(0.1, 1.0), modes)

    def go(s):
        k = []
        for i in range(12):
            s.step(1 + i % 6)
            k.append(s.run_to(s.time()[0] + (0.3 + i) / N)[1])
            k.append(tuple(s.conservation()))
        return k
    pair(sv, P, N, U0, go)


def test_stops_when_a_cell_fails(sv):
    """A run whose state goes non-physical stops at the same step with the same
    state, flags and step count, on a grid of several blocks."""
    N = 3000
    x = inputs.cell_centres(N, 1.0)
    U0 = inputs.prim_to_cons(1.4, np.ones(N), [np.where(x < 0.5, -3.0, 3.0)], np.full(N, 1e-2),
                             np.full(N, 0.5))
    r = pair(sv, sv.Params(precision=sv.FP32, tau0=0.2), N, U0,
             lambda s: s.run_to(0.05, check=False)[0])
    assert r[3] != 0 and r[5] in (sv.SV_ENONPHYS, sv.SV_EDT)


def test_captured_run_replays(sv):
    """A run captured in a CUDA graph and replayed: every replay is a launch
    of its own to the exchange words."""
    torch = pytest.importorskip("torch")
    N = 20000
    P = sv.Params(precision=sv.FP32, tau0=0.3)
    U0 = inputs.random_states(1, N, seed=1, smooth=True)
    st = torch.cuda.Stream()
    with sv.Solver(P, (N,), (1.0,), stream=st) as s:
        s.write_state(U0)
        s.step(3)
        s.write_state(U0)
        st.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            s.step(3)
        for _ in range(8):
            g.replay()
        torch.cuda.synchronize()
        U, t = s.read_state()
    with sv.Solver(P, (N,), (1.0,)) as r:
        r.set_launch(sv.LAUNCH_PER_STEP)
        r.write_state(U0)
        r.step(24)
        V, tr = r.read_state()
    assert t == tr and np.array_equal(U, V)


@pytest.mark.parametrize("prec", ["FP32", "FP32_P64", "FP64"])
@pytest.mark.parametrize("n", [1, 2, 3, 60, 61, 112, 113, 720, 721, 1791, 1792, 1793, 9599, 9600, 9601])
def test_noalloc_sizes(sv, n, prec):
    """The allocation-free step, one launch on grids a cluster holds (9600 cells
    in float, 1792 in double), against the solver's step."""
    torch = pytest.importorskip("torch")
    P = sv.Params(precision=getattr(sv, prec), tau0=0.3)
    U0 = inputs.random_states(1, n, seed=n, smooth=n > 3)
    with sv.Solver(P, (n,), (1.0,)) as s:
        s.set_launch(sv.LAUNCH_PER_STEP)
        s.write_state(U0)
        s.step(1)
        U, t = s.read_state()
        flags = s.status()
    a = torch.tensor(U0, dtype=torch.float64 if prec == "FP64" else torch.float32, device="cuda")
    b = torch.zeros_like(a)
    dt, fl = sv.step1d_noalloc(P, n, 1.0, a.data_ptr(), b.data_ptr())
    assert dt == t and fl == flags
    assert np.array_equal(b.double().cpu().numpy(), U)


@pytest.mark.parametrize("n", [500, 20000])
def test_noalloc_nonphysical_input(sv, n):
    """A state whose dt cannot be formed: no step is taken, dt 0, the flags say so."""
    torch = pytest.importorskip("torch")
    P = sv.Params(precision=sv.FP32)
    U0 = inputs.random_states(1, n, seed=n, smooth=True)
    U0[0, n // 2] = -1.0
    a = torch.tensor(U0, dtype=torch.float32, device="cuda")
    b = torch.zeros_like(a)
    dt, fl = sv.step1d_noalloc(P, n, 1.0, a.data_ptr(), b.data_ptr())
    assert dt == 0.0 and fl & sv.FLAG_NONPHYS
    assert not b.any()
