"""The fraction of a double-double number and its 128-bit fixed point (the GW
delay's and the propagation phase's coefficients, mod 1), compiled for the
host, against rational arithmetic: to 2^-104, a few units of a double-double
below one, for either sign and any size, and just beside integers.  (A
coefficient off by 2^-54 is 60 cycles off at bin 2^15 of the quartic phase.)"""
import ctypes as C
from fractions import Fraction as F

import numpy as np
import pytest

import host


def dd(x):
    """(hi, lo) of a rational number."""
    hi = float(x)
    return hi, float(x - F(hi))


def check(hi, lo):
    out = (C.c_ulonglong * 2)()
    f = host.load("dd_host").frac_fx128
    f.argtypes = [C.c_double, C.c_double, C.c_void_p]
    f(hi, lo, out)
    got = F(int(out[0]) * 2 ** 64 + int(out[1]), 2 ** 128)
    err = (got - (F(hi) + F(lo))) % 1
    assert min(err, 1 - err) <= F(1, 2 ** 104), (hi, lo, float(min(err, 1 - err)))


@pytest.mark.parametrize("scale", [1e-30, 1e-17, 1e-9, 1e-3, 0.3, 1.0, 10.0, 1e5, 1e9, 1e13])
def test_random(scale):
    g = np.random.default_rng(17)
    for _ in range(200):
        check(*dd(F(float(g.normal(0, scale))) * (1 + F(float(g.normal()) * 2.0 ** -60))))


def test_beside_integers():
    for n in (-3, -1, 0, 1, 2, 1 << 40):
        for eps in (0.0, 1e-40, 1e-20, 2.0 ** -54, 2.0 ** -53, 1e-10, 0.25, 0.5):
            for s in (-1, 1):
                check(*dd(F(n) + s * F(eps)))
