"""CPU tests of the limb-string sums, conversions, quotient and Hermite weights
(csrc/ht_mpi_ops.cuh) against exact rationals."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
RB, TWO = 29, Fraction(2)


@pytest.fixture(scope="module")
def ops(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("ops") / "libops_shim.so")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-o", out, os.path.join(HERE, "ops_shim.cpp")])
    lib = ctypes.CDLL(out)
    P, I = ctypes.c_void_p, ctypes.c_int
    lib.ops_add_sub.argtypes = [I, ctypes.c_int64, P, P, P, P]
    lib.ops_to_fz.argtypes = [I, ctypes.c_int64, P, P, I, P]
    lib.ops_hermite.argtypes = [ctypes.c_int64, P, P, P, P]
    lib.ops_hermite.restype = None
    return lib


def _value(f, limbs):
    return sum(Fraction(int(v)) * TWO ** (RB * k) for k, v in enumerate(limbs)) * TWO ** int(f)


def _parts(z, W):
    return _value(z[0], z[1:1 + W]), _value(z[0], z[1 + W:1 + 2 * W])


def _check_form(z, W):
    for c in (z[1:1 + W], z[1 + W:1 + 2 * W]):
        assert np.all(c[:-1] >= 0) and np.all(c[:-1] < (1 << RB)) and abs(int(c[-1])) < (1 << 28), z


def _strings(rng, n, W):
    """Strings in the routines' form: digits below 2^29, the top limb signed
    below 2^28; some real, some zero, some of a single limb."""
    z = np.zeros((n, 2 * W + 1), dtype=np.int32)
    z[:, 1:] = rng.integers(0, 1 << RB, (n, 2 * W))
    for c in (W, 2 * W):
        z[:, c] = rng.integers(-(1 << 28) + 1, 1 << 28, n)
    z[:, 0] = rng.integers(-300, -100, n)
    z[::7, 1 + W:] = 0
    z[::11, 1:W] = 0
    z[::13, 1 + W:2 * W] = 0
    z[5::17, 1:] = 0
    return z


@pytest.mark.parametrize("W", [5, 8])
def test_sums_and_differences(ops, W):
    """a + b and a - b: near and far apart, equal up to the last limbs (nearly
    total cancellation), opposite, and zero.  A term loses at most 2^(1 - 29 W)
    of the larger one, and the result is cut to W limbs from its highest, 2^(1
    - 29 (W - 1)) of itself."""
    rng = np.random.default_rng(40 + W)
    n = 600
    a, b = _strings(rng, n, W), _strings(rng, n, W)
    b[:, 0] = a[:, 0] + rng.integers(-40, 40, n)
    b[::5, 0] = a[::5, 0] + rng.integers(-RB * W - 5, RB * W + 5, len(b[::5]))
    for q in range(0, n, 6):  # the same number but for its lowest limbs
        b[q] = a[q]
        low = rng.integers(0, W)
        b[q, 1:1 + low] = rng.integers(0, 1 << RB, low)
    b[3::24] = a[3::24]
    s, d = np.zeros_like(a), np.zeros_like(a)
    ptr = lambda v: v.ctypes.data
    assert ops.ops_add_sub(W, n, ptr(a), ptr(b), ptr(s), ptr(d)) == 0
    for q in range(n):
        x, y = _parts(a[q], W), _parts(b[q], W)
        big = max(abs(v) for v in x + y)
        for out, sign in ((s[q], 1), (d[q], -1)):
            _check_form(out, W)
            want, got = [u + sign * v for u, v in zip(x, y)], _parts(out, W)
            size = max(abs(v) for v in want)
            for w, g in zip(want, got):
                assert abs(w - g) <= TWO ** (2 - RB * W) * big + TWO ** (1 - RB * (W - 1)) * size, (q, sign)


@pytest.mark.parametrize("W", [5, 8])
def test_fixed_point_to_string(ops, W):
    """The window of W limbs of a fixed-point string from the highest
    significant limb of either component: strings with 0 to all of their upper
    limbs empty, of either sign, -2^(29 k) (whose limb k is all sign), and
    zero.  One unit of the string's last limb, which normalising may shift."""
    WA = W + 1
    rng = np.random.default_rng(60 + W)
    rows = []
    for top in range(WA):
        for _ in range(12):
            r = np.zeros((2, WA), dtype=np.int64)
            r[:, :top + 1] = rng.integers(0, 1 << RB, (2, top + 1))
            for c in (0, 1):
                if rng.random() < 0.5:  # negative: the digits above are all ones, the top limb -1
                    r[c, top + 1:] = (1 << RB) - 1
                    if top + 1 < WA:
                        r[c, -1] = -1
                    else:
                        r[c, -1] = -int(r[c, -1] >> 2) - 1
                elif top + 1 == WA:
                    r[c, -1] >>= 2
            rows.append(r)
        for c in (0, 1):  # -2^(29 top), the other component zero
            r = np.zeros((2, WA), dtype=np.int64)
            r[c, top:] = (1 << RB) - 1
            r[c, -1] = -1
            rows.append(r)
    rows.append(np.zeros((2, WA), dtype=np.int64))
    n, F = len(rows), -117
    ar = np.ascontiguousarray([r[0] for r in rows], dtype=np.int32)
    ai = np.ascontiguousarray([r[1] for r in rows], dtype=np.int32)
    out = np.zeros((n, 2 * W + 1), dtype=np.int32)
    assert ops.ops_to_fz(W, n, ar.ctypes.data, ai.ctypes.data, F, out.ctypes.data) == 0
    for q in range(n):
        _check_form(out[q], W)
        want = (_value(F, ar[q]), _value(F, ai[q]))
        size = max(abs(v) for v in want)
        for w, g in zip(want, _parts(out[q], W)):
            assert abs(w - g) <= TWO ** int(out[q, 0])
        if size:  # the window starts at the highest significant limb
            assert TWO ** int(out[q, 0]) <= size * TWO ** (2 - RB * (W - 1))
        else:
            assert not np.any(out[q, 1:])


def test_quotients_and_hermite_weights(ops):
    """u = (t1 - s0) / (s1 - s0) and the four weights for steps of the tracker:
    intervals from 1e-12 to 0.1, predictions inside and far beyond them, t
    close to 1 and to 0, differences as exact quad doubles.  A string keeps at
    least 29 * 7 + 1 bits: the quotient's three Newton steps and product stay
    within 16 units of 2^-203, a weight within 32 of the sum of its terms'
    moduli."""
    rng = np.random.default_rng(5)
    n = 400
    s0 = rng.random(n)
    s1 = s0 + 10.0 ** rng.uniform(-12, -1, n)
    t1 = s1 + (s1 - s0) * 10.0 ** rng.uniform(-6, 3, n)
    s0[:20] = 1.0 - 2.0 ** -30 * rng.random(20)
    s1[:20] = 1.0 - 2.0 ** -40 * rng.random(20)
    t1[:20] = 1.0
    s0[20:30], s1[20:30], t1[20:30] = 0.0, 0.05, 0.125
    t1[30:40] = s0[30:40] + 0.5 * (s1[30:40] - s0[30:40])

    def diff(x, y):  # the two doubles of x - y
        out = np.zeros((n, 4))
        out[:, 0] = x - y
        out[:, 1] = [float(Fraction(float(p)) - Fraction(float(q)) - Fraction(float(h)))
                     for p, q, h in zip(x, y, out[:, 0])]
        return out

    a, b = diff(t1, s0), diff(s1, s0)
    quo, w = np.zeros((n, 9), dtype=np.int32), np.zeros((n, 4, 9), dtype=np.int32)
    ops.ops_hermite(n, a.ctypes.data, b.ctypes.data, quo.ctypes.data, w.ctypes.data)
    unit = TWO ** -203
    for q in range(n):
        num = sum(Fraction(float(v)) for v in a[q])
        d = sum(Fraction(float(v)) for v in b[q])
        u = num / d
        assert abs(_value(quo[q, 0], quo[q, 1:]) - u) <= 16 * unit * abs(u), q
        terms = [(2 * u ** 3, -3 * u ** 2, Fraction(1)), (u ** 3 * d, -2 * u ** 2 * d, u * d),
                 (-2 * u ** 3, 3 * u ** 2), (u ** 3 * d, -u ** 2 * d)]
        for k in range(4):
            got = _value(w[q, k, 0], w[q, k, 1:])
            # (u's own error passes to the weight through the terms: at most three times each)
            assert abs(got - sum(terms[k])) <= (32 + 3 * 16) * unit * sum(abs(v) for v in terms[k]), (q, k)
