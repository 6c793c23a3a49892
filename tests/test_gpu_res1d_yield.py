"""Long runs of the resident 1D step loop leave the GPU to other streams now and
then: its launches fill every SM, so a launch may not last for the whole run."""
import time

import pytest

from gpu_util import need_gpu
from paper_1805_03442_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec, N, k", [("FP32", 182400, 65536), ("FP64", 34048, 16384)])
def test_other_streams_run_meanwhile(prec, N, k):
    sv = need_gpu()
    torch = pytest.importorskip("torch")
    P = sv.Params(precision=getattr(sv, prec), tau0=float("inf"), S=0.0)
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    x = torch.zeros(1024, device="cuda")
    with sv.Solver(P, (N,), (1.0,), stream=mine) as s:
        s.write_state(inputs.waves_1d(1.4, N, 1.0, inputs.equilibrium_primitive(0.1, 0.0), []))
        s.step(2)
        with torch.cuda.stream(other):
            x.add_(1.0)
        torch.cuda.synchronize()
        s.step(k)                                # 0.3 s and more
        end = torch.cuda.Event()
        end.record(mine)
        time.sleep(0.05)
        assert not end.query()
        with torch.cuda.stream(other):
            x.add_(1.0)
        other.synchronize()
        assert not end.query()                   # the run is still going on
        torch.cuda.synchronize()
        assert s.time()[1] == k + 2 and s.status() == 0


def test_run_to_over_several_launches():
    """A run to a time beyond one launch's steps, and to the step cap inside one."""
    sv = need_gpu()
    N = 3000
    P = sv.Params(precision=sv.FP32, tau0=float("inf"), S=0.0)
    modes = inputs.random_phase_modes(2, inputs.acoustic_shape(1.4), 4, 1, 1e-3)
    U0 = inputs.waves_1d(1.4, N, 1.0, inputs.equilibrium_primitive(0.1, 0.0), modes)
    out = []
    for mode in (sv.LAUNCH_PER_STEP, sv.LAUNCH_AUTO, sv.LAUNCH_PERSISTENT):
        with sv.Solver(P, (N,), (1.0,)) as s:
            s.set_launch(mode)
            s.write_state(U0)
            got = [s.run_to(0.3), s.time(), s.run_to(0.9, max_steps=1500, check=False), s.time()]
            out.append(got + [s.read_state()[0].tobytes()])
    assert out[0][0][1] > 2048 and out[0][2] == (sv.SV_EMAXSTEPS, 1500)
    assert out[1] == out[0] and out[2] == out[0]
