"""The batched sweep's window kernel (csrc/sv_batch_kernel.cuh) at the edges of
its decomposition, against single solvers stepped launch by launch, bit for bit:
sizes around whole windows (60 cells in float, 28 in double) and around what one
round of a cluster holds, with few runs (a cluster per run) and with many (one
block per run), and runs read back before, between and after launches."""
import numpy as np
import pytest

from gpu_util import need_gpu
from paper_1805_03442_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    return need_gpu()


class Run:
    def __init__(self, n, i, steps):
        self.n, self.L, self.m = n, 1.0, 1
        self.S, self.tau0 = 0.5, 0.3 + 0.1 * (i % 3)
        self.tau_rho, self.tau_T = -1.0, -1.5
        self.Q_rho, self.Q_T, self.I_rho, self.I_T = (0.0, 0.0, 0.0, 0.0) if i % 2 else (0.5, 0.3, -0.2, 0.1)
        self.t_end = steps * 0.4 / n / 2.0


def single(sv, prec, run, U0):
    P = sv.Params(precision=prec, S=run.S, tau0=run.tau0, tau_rho=run.tau_rho, tau_T=run.tau_T,
                  Q_rho=run.Q_rho, Q_T=run.Q_T, I_rho=run.I_rho, I_T=run.I_T)
    with sv.Solver(P, (run.n,), (run.L,)) as s:
        s.set_launch(sv.LAUNCH_PER_STEP)
        s.write_state(U0)
        _, k = s.run_to(run.t_end, check=False)
        U, t = s.read_state()
        return U, t, k, s.status()


SIZES = {"FP32": [1, 2, 3, 59, 60, 61, 119, 479, 480, 481, 3839, 3840, 3841, 7681],
         "FP64": [1, 2, 3, 27, 28, 29, 223, 224, 225, 1793]}


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("copies", [1, 45])
def test_sizes(sv, prec, copies):
    p = getattr(sv, prec)
    runs = [Run(n, i, 12) for i, n in enumerate(SIZES[prec])]
    states = [inputs.random_states(1, r.n, seed=r.n, smooth=r.n > 3) * 1.0 for r in runs]
    want = [single(sv, p, r, U) for r, U in zip(runs, states)]
    with sv.Batch(sv.Params(precision=p), runs * copies, states * copies, log_cap=5) as b:
        for i in (0, len(runs) - 1):          # before the first launch: what was uploaded
            U, t, k, f = b.read(i)
            assert t == 0.0 and k == 0 and f == 0
        for _ in range(2):
            b.run()
            for i in range(len(runs) * copies):
                U, t, k, f = b.read(i)
                w = want[i % len(runs)]
                assert np.array_equal(U, w[0], equal_nan=True), runs[i % len(runs)].n
                assert (t, k, f) == w[1:]
                tl, a = b.mode_log(i)
                assert len(tl) >= 2 and tl[0] == 0.0 and tl[-1] == t
                v = U[1] / U[0]
                x = (np.arange(len(v)) + 0.5) / len(v)
                amp = np.mean(v * np.exp(-2j * np.pi * x))
                assert abs(a[-1] - amp) <= 1e-5
            b.reset(states * copies)
