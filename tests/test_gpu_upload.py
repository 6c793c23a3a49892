"""Upload and download of a state (one kernel each): the four-cells-at-a-time form
and the element form around the sizes where one takes over from the other, the
dt that the upload leaves, and the state read back.

Tolerances.  The state: exact for the float and double layouts; the
perturbation layout rounds U - U_ref to float, 2^-24 of it.  dt: float, ten
roundings of 2^-24 in c (p amplifies those of E and E_nu at most threefold here)
and 2^-22 from each logarithm of tau, below 4e-6 together; double 1e-13."""
import numpy as np
import pytest

from gpu_util import need_gpu
from oracle import orc as O
from paper_1805_03442_gb300 import inputs

pytestmark = pytest.mark.gpu

SIZES = [(1,), (2,), (3,), (4,), (5,), (1020,), (1023,), (1024,), (622592,), (622597,), (622600,),
         (64, 33), (63, 31), (16, 8, 6), (9, 7, 5)]


@pytest.fixture(scope="module")
def sv():
    return need_gpu()


@pytest.mark.parametrize("prec", ["FP32", "FP32_PC", "FP32_PS", "FP64"])
@pytest.mark.parametrize("host", ["float32", "float64"])
@pytest.mark.parametrize("n", SIZES)
def test_upload_download_and_dt(sv, prec, host, n):
    torch = pytest.importorskip("torch")
    dim, cells = len(n), int(np.prod(n))
    U = inputs.random_states(dim, cells, seed=cells).reshape(dim + 3, cells).astype(host)
    wide = host == "float64"
    P = sv.Params(precision=getattr(sv, prec), tau0=0.3)
    got = []
    for offset in (0, 1):                   # 16-byte aligned, and not
        hin = torch.empty(U.size + 1, dtype=getattr(torch, host), pin_memory=True)[offset:][:U.size]
        hout = torch.empty(U.size + 1, dtype=getattr(torch, host), pin_memory=True)[offset:][:U.size]
        hin.copy_(torch.from_numpy(U.reshape(-1)))
        with sv.Solver(P, n) as s:
            (s.write_state_ptr if wide else s.write_state_ptr_f32)(hin.data_ptr())
            dt = s.dt()
            (s.read_state_ptr if wide else s.read_state_ptr_f32)(hout.data_ptr())
            back, _ = s.read_state()        # pageable, double
            assert s.status() == 0
        got.append((dt, hout.numpy().reshape(U.shape).copy(), back.reshape(U.shape)))
    (dt, out, back), (dt1, out1, back1) = got
    assert dt == dt1 and np.array_equal(out, out1) and np.array_equal(back, back1)
    exact = U.astype(np.float64)
    if prec == "FP32_PS":
        ref = np.zeros((dim + 3, 1))
        ref[0], ref[-2], ref[-1] = 1.0, 1.0 / (P.gamma - 1.0) + P.Ck + P.S, P.Ck + P.S
        assert np.all(np.abs(back - exact) <= 1.01 * 2.0 ** -24 * np.abs(exact - ref) + 4e-15)
    else:
        assert np.array_equal(back, exact if prec == "FP64" else U.astype(np.float32).astype(np.float64))
    assert np.array_equal(out, back.astype(host))
    Po = O.Params(tau0=0.3)
    want = O.dt_cfl(Po, back, n if dim > 1 else n[0], 1.0 / n[0])
    assert abs(dt / want - 1.0) <= (1e-13 if prec == "FP64" else 4e-6)
