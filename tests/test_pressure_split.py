"""The pressure recovery of SV_FP32_P64 and SV_FP32_PC (eq. 5 of float operands
without a rounding before the last, csrc/sv_model.cuh pressure<float, 2>),
emulated in numpy float32 with a double-exact fused multiply-add, against the
subtraction carried out in double.  The two may differ by the last bit of p:
one rounding to float each, of values at most 2^-47 apart, so by one ulp where
that gap straddles a float midpoint."""
import numpy as np
import pytest

f32, f64 = np.float32, np.float64
G1 = 0.4
G1H = f32(G1)
G1L = f32(G1 - f64(G1H))


def fma(a, b, c):
    """round(a b + c) to float: the product of two floats is exact in double,
    its sum with c rounds in double first (2^-53, far below a float ulp)."""
    return (a.astype(f64) * b.astype(f64) + np.asarray(c, f64)).astype(f32)


def split(kin2, E, Ev):
    h = f32(0.5) * kin2
    s = E - Ev
    e1 = (E - s) - Ev
    t = s - h
    e2 = (s - t) - h
    g1, lo = np.full_like(t, G1H), np.full_like(t, G1L)
    return fma(g1, t, fma(lo, t, g1 * (e1 + e2)))


def states(seed, ev, n=200000):
    rng = np.random.default_rng(seed)
    kin2 = (10.0 ** rng.uniform(-12, 2, n) * rng.integers(0, 2, n)).astype(f32)
    Ev = (ev * rng.uniform(0.5, 2.0, n)).astype(f32)
    p = rng.uniform(1e-3, 4.0, n)
    E = (p / 0.4 + 0.5 * kin2 + Ev).astype(f32)
    return kin2, E, Ev


@pytest.mark.parametrize("ev", [0.0, 0.1, 1.0, 30.0, 1000.0, 1e5])
def test_split_is_the_double_subtraction_to_its_last_bit(ev):
    kin2, E, Ev = states(int(ev) + 1, ev)
    # E_nu = 1e5 leaves some of these states without pressure (p <= 0): there
    # only the sign of p is used, the next test's matter
    ok = E.astype(f64) - 0.5 * kin2.astype(f64) - Ev.astype(f64) > 0
    assert ok.mean() > 0.9
    kin2, E, Ev = kin2[ok], E[ok], Ev[ok]
    q = E.astype(f64) - 0.5 * kin2.astype(f64) - Ev.astype(f64)
    want, got = (G1 * q).astype(f32), split(kin2, E, Ev)
    ulp = np.spacing(np.abs(want))
    assert np.all(np.abs(got.astype(f64) - want.astype(f64)) <= ulp)
    # against 64 bits: as close as the double policy's own rounding to float
    err = np.abs(got.astype(f64) - G1 * q)
    assert np.all(err <= (0.5 + 2.0 ** -20) * ulp)


def test_sign_of_p_is_exact():
    """States around and below p = 0, where the guard decides on the sign."""
    rng = np.random.default_rng(9)
    n = 400000
    Ev = (10.0 ** rng.uniform(-3, 3, n)).astype(f32)
    h = 10.0 ** rng.uniform(-6, 3, n)
    E = (Ev + h * rng.choice([0.0, 0.5, 1.0, 1.0 + 1e-7, 1.0 - 1e-7, 2.0], n)).astype(f32)
    E = np.where(rng.random(n) < 0.1, (0.9 * Ev).astype(f32), E)
    kin2 = (2.0 * h).astype(f32)
    q = E.astype(f64) - 0.5 * kin2.astype(f64) - Ev.astype(f64)
    assert np.array_equal(np.sign(split(kin2, E, Ev)), np.sign(q))
