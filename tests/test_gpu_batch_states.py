"""States of the batched sweep read back through the page-locked copy of all of
them, and run by run where they are too many for it (64 MB): the same runs give
the same states, times and steps bit for bit, before a launch, after it and after
a second upload."""
import numpy as np
import pytest

from gpu_util import need_gpu
from paper_1805_03442_gb300 import inputs

pytestmark = pytest.mark.gpu


class Run:
    def __init__(self, n, t_end):
        self.n, self.L, self.m, self.t_end = n, 1.0, 1, t_end
        self.S, self.tau0, self.tau_rho, self.tau_T = 0.5, 0.3, -1.0, -1.5
        self.Q_rho = self.Q_T = self.I_rho = self.I_T = 0.0


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
def test_states_within_and_beyond_the_copy(prec):
    sv = need_gpu()
    P = sv.Params(precision=getattr(sv, prec))
    small = [Run(n, 7 * 0.4 / n / 2.0) for n in (1, 33, 601, 1024)]
    big = Run((64 << 20) // 16, 0.0)             # alone as large as the copy may be
    first = [inputs.random_states(1, r.n, seed=r.n) for r in small]
    other = [inputs.random_states(1, r.n, seed=r.n + 1) for r in small]
    U = np.repeat([[1.0], [0.0], [3.6], [1.1]], big.n, axis=1)
    with sv.Batch(P, small, first, log_cap=3) as a, sv.Batch(P, small + [big], first + [U], log_cap=3) as b:
        for states in (first, other):
            a.reset(states)
            b.reset(states + [U])
            for launch in (False, True):
                if launch:
                    a.run()
                    b.run()
                for i, r in enumerate(small):
                    (x, *xs), (y, *ys) = a.read(i), b.read(i)
                    assert xs == ys and np.array_equal(x, y)
                    if launch:
                        assert xs[0] == r.t_end
                    else:
                        assert np.array_equal(x, states[i] if prec == "FP64" else states[i].astype(np.float32))
        assert np.array_equal(b.read(len(small))[0], U if prec == "FP64" else U.astype(np.float32))
