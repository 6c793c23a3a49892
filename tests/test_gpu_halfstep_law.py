"""The power laws of eq. 6 at a half-step state past p = 0 (heated within half a
step): a whole power of a negative temperature is a number, in double as in the
oracle, also where the density's exponent is a half one."""
import numpy as np
import pytest

from gpu_util import need_gpu, oracle_params
from oracle import orc as O
from paper_1805_03442_gb300 import inputs

pytestmark = pytest.mark.gpu

LAWS = [dict(tau_rho=-0.5, tau_T=-1.0), dict(tau_rho=-1.5, tau_T=-2.0), dict(tau_rho=0.5, tau_T=1.0),
        dict(tau_rho=-3.5, tau_T=-1.0), dict(tau_rho=-0.5, tau_T=2.0), dict(tau_rho=-1.0, tau_T=-1.0),
        dict(tau_rho=-0.5, tau_T=-1.0, Q_rho=0.5, Q_T=1.0, I_rho=-2.5, I_T=-2.0)]


@pytest.mark.parametrize("law", LAWS)
@pytest.mark.parametrize("n", [(60,), (20000,), (24, 10), (8, 6, 5)])
def test_uniform_heated_state(law, n):
    """Uniform cells, so a step is the source alone: E_nu = 0.17 of E = 2.67 heated
    to about 3.4 in half a step, T = -0.17."""
    sv = need_gpu()
    h = 1.0 / n[0]
    rho = 1.7
    half = 0.2 * h / np.sqrt(1.4 / rho)          # dt / 2 of cfl 0.4 at rest
    P = sv.Params(precision=sv.FP64, tau0=1.0, c_tau=1e9, S=3.2 / half / rho, **law)
    one = np.ones(int(np.prod(n)))
    U0 = inputs.prim_to_cons(1.4, rho * one, [0 * one] * len(n), one, 0.1 * one)
    Po = oracle_params(P)
    nn = n if len(n) > 1 else n[0]
    ref, _ = O.step(Po, U0, nn, h, O.dt_cfl(Po, U0, nn, h))
    assert np.all(np.isfinite(ref))
    with sv.Solver(P, n, tuple(m / n[0] for m in n)) as s:
        for mode in (sv.LAUNCH_PER_STEP, sv.LAUNCH_AUTO):
            s.set_launch(mode)
            s.write_state(U0)
            s.step(1)
            U, _ = s.read_state()
            U = U.reshape(ref.shape)
            assert np.max(np.abs(U - ref) / np.maximum(np.abs(ref), 1.0)) < 1e-12
