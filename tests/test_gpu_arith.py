"""The step kernels' own arithmetic, function by function on the device
(tests/arith_probe.cu): the reciprocal and square root of the double kernels
(csrc/sv_f64.cuh) against the exact results, with the bound that the series gives."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


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
