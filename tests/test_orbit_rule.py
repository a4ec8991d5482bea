"""The orbit solver's stopping rule, compiled for the host, on sequences of
updates whose contraction is known: an accepted orbit has at most one ulp of v
(2.2e-16) left, whatever the contraction; the usual ones are accepted after
three evaluations, and updates that are not numbers never are."""
import ctypes as C
import math

import numpy as np
import pytest

import host


@pytest.fixture(scope="module")
def rule():
    lib = host.load("orbit_rule_host")
    lib.again.argtypes = [C.c_float] * 2
    lib.settled.argtypes = [C.c_float] * 3
    return lib


def solve(rule, u1, rho):
    """(accepted, evaluations, error left) for updates u1, u1 rho, ..."""
    u = [u1 * rho ** k for k in range(6)]
    if not rule.again(u[0], u[1]):
        return rule.settled(u[0], u[1], u[2]), 3, u[3]
    return rule.settled(u[1], u[2], u[3]), 4, u[4]


def test_accepted_orbits_are_settled(rule):
    n = 0
    for u1 in np.logspace(-9, -3, 61):
        for rho in np.logspace(-6, -0.5, 111):
            ok, _, left = solve(rule, u1, rho)
            n += bool(ok)
            assert not ok or left <= 2.0 ** -52, (u1, rho, left)
    assert n > 1000


@pytest.mark.parametrize("u1,rho", [(1e-7, 5e-5), (1e-6, 2e-4), (1e-6, 1e-4), (3e-7, 3e-4), (5e-6, 2e-5)])
def test_usual_orbits_take_three(rule, u1, rho):
    ok, evaluations, _ = solve(rule, u1, rho)
    assert ok and evaluations == 3


def test_rounding_level_and_nan(rule):
    assert not rule.again(1e-6, 1e-16) and rule.settled(1e-6, 1e-16, 9e-17) and rule.settled(0.0, 0.0, 0.0)
    for bad in (math.nan, math.inf):
        assert rule.again(1e-6, bad)
        assert not rule.settled(1e-6, 1e-10, bad)
    assert not rule.settled(1e-6, math.nan, 1e-14)
