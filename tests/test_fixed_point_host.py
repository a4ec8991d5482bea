"""The FP64 waveform kernel's fixed-point arithmetic, compiled for the host:
sines and cosines, harmonic sums and response may be no further from long
double than the same steps in double, in rms and at worst -- over random and
boundary phases, over the amplitudes of circular to eccentric orbits and over
the drifts of e within a segment from far inside an inspiral to its last hours
(one and two words for the quadratic coefficients).
"""
import ctypes as C

import numpy as np
import pytest

import host

scipy_special = pytest.importorskip("scipy.special")


def ptr(a):
    return a.ctypes.data_as(C.c_void_p)


def phases(g, count):
    """Random phases, and the ones beside the multiples of 1/1024 and 1/2048 of a cycle."""
    p = g.integers(0, 1 << 64, count, dtype=np.uint64)
    p[: count // 8] = (g.integers(0, 2048, count // 8, dtype=np.uint64) << np.uint64(53)) + \
        g.integers(-2, 3, count // 8).astype(np.uint64)
    return p


def no_worse(fixed, dbl, what=None):
    rms, most = [[f(x) for x in (fixed, dbl)] for f in (lambda x: np.sqrt(np.mean(x ** 2)), lambda x: np.abs(x).max())]
    assert rms[0] <= rms[1] and most[0] <= most[1], (what, rms, most)


def test_sincos():
    p = phases(np.random.default_rng(1), 1 << 16)
    fixed, dbl = np.zeros((len(p), 2)), np.zeros((len(p), 2))
    host.load("wave_fixed_host").sincos_errors(ptr(p), len(p), ptr(fixed), ptr(dbl))
    no_worse(fixed, dbl)


def amplitudes(n_max, e):
    """a_n, b_n, c_n of the Peters-Mathews sums at eccentricity e, [n_max, 3]."""
    n = np.arange(1, n_max + 1)
    j = {k: scipy_special.jv(n + k, n * e) for k in (-2, -1, 0, 1, 2)}
    a = n * (j[-2] - 2 * e * j[-1] + 2 / n * j[0] + 2 * e * j[1] - j[2])
    b = n * np.sqrt(1 - e * e) * (j[-2] - 2 * j[0] + j[2])
    return np.stack([a, b, 2 * j[0]], axis=1)


@pytest.mark.parametrize("n_max", [5, 20, 32])
def test_harmonic_sums(n_max):
    lib = host.load("wave_fixed_host")
    g = np.random.default_rng(n_max)
    count, words = 4096, set()
    for e in (0.01, 0.1, 0.2, 0.3, 0.5, 0.7, 0.9):
        for drift in (1e-6, 1e-5, 1e-4, 3e-4, 1e-3, 3e-3):   # e falls by this in a segment
            f = [amplitudes(n_max, e - drift * t) for t in (0.0, 0.5, 1.0)]
            q = np.ascontiguousarray(np.stack(
                [f[0], -3 * f[0] + 4 * f[1] - f[2], 2 * f[0] - 4 * f[1] + 2 * f[2]], axis=2))   # [n][quantity][power]
            s = np.abs(q).sum(axis=(0, 1))
            if 32 * s[1] >= s[0]:
                continue                # in double in the kernel too
            p, r = phases(g, count), g.integers(0, 1024, count).astype(np.int32)
            fixed, dbl = np.zeros((count, 3)), np.zeros((count, 3))
            words.add(lib.harmonic_errors(ptr(q), n_max, ptr(p), ptr(r), count, ptr(fixed), ptr(dbl)))
            no_worse(fixed, dbl, (e, drift))
    assert words == {0, 1}


def test_response():
    lib = host.load("wave_fixed_host")
    g = np.random.default_rng(3)
    for _ in range(8):
        # orthonormal orbital-plane vectors as the prologue projects them on the sky basis
        q, _ = np.linalg.qr(g.standard_normal((3, 3)))
        e1, e2, S = q.T
        lam = np.arccos(g.uniform(-1, 1))
        w, _ = np.linalg.qr(g.standard_normal((3, 3)))
        P, Q = w[:, 0], w[:, 1]
        cl, sl = np.cos(lam), np.sin(lam)
        geo = np.array([P @ e1, P @ e2, Q @ e1, Q @ e2, cl * (P @ e1), cl * (P @ e2), cl * (Q @ e1), cl * (Q @ e2),
                        sl * (P @ S), sl * (Q @ S)])
        count = 4096
        gm, al = phases(g, count), phases(g, count)
        sums = (g.uniform(-1, 1, (count, 3)) * 2.0 ** 60).astype(np.int64)
        fixed, dbl = np.zeros((count, 2)), np.zeros((count, 2))
        lib.response_errors(ptr(geo), ptr(gm), ptr(al), ptr(sums), count, ptr(fixed), ptr(dbl))
        no_worse(fixed, dbl)
