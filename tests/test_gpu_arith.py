"""The step kernels' own arithmetic, function by function on the device
(tests/arith_probe.cu): the reciprocal and square root of the double kernels
(csrc/sv_f64.cuh) and the pressure recovery of SV_FP32_P64 / SV_FP32_PC
(pressure<2> of csrc/sv_model.cuh, packed in csrc/sv_pair1d.cuh), each against
64 bits with the bound that its series or its sums give."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
f32, f64 = np.float32, np.float64


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    need_gpu()
    so = str(tmp_path_factory.mktemp("probe") / "arith_probe.so")
    root = os.path.dirname(HERE)
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                    "-Xcompiler", "-fPIC", "-I" + os.path.join(root, "include"),
                    "-I" + os.path.join(root, "paper_1805_03442_gb300", "csrc"), "-o", so,
                    os.path.join(HERE, "arith_probe.cu")], check=True)
    return ctypes.CDLL(so)


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def f64_op(probe, op, x):
    y = np.empty_like(x)
    assert probe.probe_f64(op, ptr(x), ptr(y), len(x)) == 0
    return y


def two_product(a, b):
    """a b as an unevaluated sum (Dekker's product, Veltkamp's split)."""
    def split(v):
        c = (2.0 ** 27 + 1.0) * v
        hi = c - (c - v)
        return hi, v - hi
    p = a * b
    (ah, al), (bh, bl) = split(a), split(b)
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def arguments(seed):
    """Random mantissas over the exponents of any state, and the neighbours of
    powers of two."""
    rng = np.random.default_rng(seed)
    x = np.ldexp(rng.uniform(1.0, 2.0, 4_000_000), rng.integers(-300, 301, 4_000_000))
    p = np.ldexp(1.0, np.arange(-300, 301))
    near = [p]
    lo = hi = p
    for _ in range(40):
        lo, hi = np.nextafter(lo, 0.0), np.nextafter(hi, np.inf)
        near += [lo, hi]
    return np.concatenate([x] + near)


def test_reciprocal(probe):
    """y0 (1 + e + e^2) leaves e^3 of the estimate's error e; the last operation
    rounds, and the one before it by 2^-53 of e."""
    x = arguments(1)
    p, q = two_product(x, f64_op(probe, 2, x))
    e = np.max(np.abs((1.0 - p) - q))
    assert e < 2.0 ** -18
    y = f64_op(probe, 0, x)
    p, q = two_product(x, y)
    err = np.abs((1.0 - p) - q) * y / np.spacing(y)
    print(f"estimate 2^{np.log2(e):.2f}, reciprocal {err.max():.4f} ulp")
    assert err.max() <= 0.5 + 2.0 ** 53 * e ** 3 + 2.0 ** -16


def test_square_root(probe):
    """With e = 1 - g^2 / x of the estimate's g, g + d y0 (1/2 + 3/8 d y0^2)
    leaves 5/16 e^3 of the series and 3/8 e^3 of y0^2 for 1/x."""
    x = arguments(2)
    y0 = f64_op(probe, 3, x)
    g = x * y0
    p, q = two_product(g, g)
    e = np.max(np.abs(((x - p) - q) / x))
    assert e < 2.0 ** -18
    y = f64_op(probe, 1, x)
    p, q = two_product(y, y)
    err = np.abs((x - p) - q) / (2.0 * y) / np.spacing(y)
    print(f"estimate 2^{np.log2(e):.2f}, square root {err.max():.4f} ulp")
    assert err.max() <= 0.5 + 11 / 16 * 2.0 ** 53 * e ** 3 + 2.0 ** -16


def pressures(probe, gamma, kin2, E, Ev):
    s = np.ascontiguousarray(np.stack([kin2, E, Ev]))
    p = np.empty((2, len(E)), f32)
    probe.probe_pressure.argtypes = [ctypes.c_double, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]
    assert probe.probe_pressure(gamma, ptr(s), ptr(p), len(E)) == 0
    return p


def states(seed, ev, n=400_000):
    rng = np.random.default_rng(seed)
    kin2 = (10.0 ** rng.uniform(-12, 2, n) * rng.integers(0, 2, n)).astype(f32)
    p = rng.uniform(1e-3, 4.0, n)
    Ev = ev * rng.uniform(0.5, 2.0, n)
    E = (p / 0.4 + 0.5 * kin2 + np.maximum(Ev, 0.0)).astype(f32)
    if ev < 0:                            # E_nu between -E and 0
        Ev = -E * rng.uniform(0.0, 1.0, n)
    return kin2, E, Ev.astype(f32)


@pytest.mark.parametrize("gamma", [1.4, 5 / 3, 1.05])
@pytest.mark.parametrize("ev", [-1.0, 0.0, 0.1, 1.0, 30.0, 1000.0])
def test_pressure_without_a_rounding_before_the_last(probe, gamma, ev):
    """gamma - 1 times the difference that double carries out, rounded once: what
    is rounded before is 2^-24 of e1 + e2 (themselves 2^-24 of the sums s and t)
    and of the small part of gamma - 1.  The packed recovery gives the same bits."""
    kin2, E, Ev = states(int(10 * ev) + 20, ev)
    q = E.astype(f64) - 0.5 * kin2.astype(f64) - Ev.astype(f64)
    ok = q > 0
    assert ok.mean() > 0.9
    one, two = pressures(probe, gamma, kin2, E, Ev)
    assert np.array_equal(one, two)
    want = (gamma - 1.0) * q[ok]
    ulp = np.spacing(want.astype(f32)).astype(f64)
    s = np.abs(E.astype(f64) - Ev)[ok]
    err = np.abs(one[ok].astype(f64) - want) / ulp
    assert np.all(err <= 0.5 + 2.0 ** -22 * (1.0 + s / q[ok]))
    # the double policy's own rounding of the same number: its last bit at most
    assert np.all(np.abs(one[ok].astype(f64) - want.astype(f32)) <= ulp)


def test_sign_of_p_is_exact(probe):
    """States around and below p = 0, where the guard decides on the sign."""
    rng = np.random.default_rng(9)
    n = 400_000
    Ev = (10.0 ** rng.uniform(-3, 3, n)).astype(f32)
    h = 10.0 ** rng.uniform(-6, 3, n)
    E = (Ev + h * rng.choice([0.0, 0.5, 1.0, 1.0 + 1e-7, 1.0 - 1e-7, 2.0], n)).astype(f32)
    E = np.where(rng.random(n) < 0.1, (0.9 * Ev).astype(f32), E)
    kin2 = (2.0 * h).astype(f32)
    q = E.astype(f64) - 0.5 * kin2.astype(f64) - Ev.astype(f64)
    for p in pressures(probe, 1.4, kin2, E, Ev):
        assert np.array_equal(np.sign(p), np.sign(q))
