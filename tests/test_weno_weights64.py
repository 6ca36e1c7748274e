"""The FP64 WENO5 weights in 64-bit integer arithmetic (weno_weights64.cuh, its
host build) against exact rational arithmetic.

Bound: a smoothness sum is good to 2^-54 (the cut-off bits of its three terms),
a product of four of them to 4 * 2^-54 plus a few 2^-57, a weight takes one such
product and one denominator of them, and its own rounding adds 2^-53: below
2^-51 altogether."""
import ctypes
import os
import subprocess
from fractions import Fraction as F

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2507_11542_gb300", "csrc")


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("w64") / "libweights64.so")
    subprocess.check_call(["g++", "-O2", "-ffp-contract=off", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, "-x", "c++",
                           os.path.join(HERE, "probes", "weights64_probe.cpp"), "-o", out])
    lib = ctypes.CDLL(out)
    lib.weights64_probe.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong]
    return lib


def windows(kind, rng, n):
    e = rng.normal(size=(n, 5))
    if kind == "kink":
        e[:, :2] = 1.0
        e[:, 2:] = -1.0 + 1e-9 * rng.normal(size=(n, 3))
    elif kind == "jump":
        e *= 10.0 ** rng.uniform(-14, 0, size=(n, 5))
    elif kind == "one_side_flat":
        e[:, 2:] = 0.0
    elif kind == "powers_of_two":
        e = np.ldexp(np.sign(e), rng.integers(-3, 4, size=(n, 5)))
    elif kind == "smooth":
        x, h = rng.uniform(0, 6, size=(n, 1)), 10.0 ** rng.uniform(-4, 0, size=(n, 1))
        k = np.arange(5)
        e = np.sin(x + (k + 1) * h) - np.sin(x + k * h)
    elif kind == "tiny":      # the additive floor decides
        e *= 1e-50
    elif kind == "huge":
        e *= 1e140
    return e


@pytest.mark.parametrize("kind", ["random", "kink", "jump", "one_side_flat", "powers_of_two", "smooth", "tiny", "huge"])
def test_weights_against_rationals(probe, kind):
    rng = np.random.default_rng(len(kind))
    n, floor12 = 300, 12e-99 * 0.07 ** 2
    e = windows(kind, rng, n)
    d = np.diff(e, axis=1)
    t = np.diff(d, axis=1)
    rows = np.empty((n, 7))
    rows[:, 0:3], rows[:, 3:5] = t, d[:, 1:3]
    rows[:, 5], rows[:, 6] = np.abs(e).max(axis=1), floor12
    got = np.empty((n, 4))
    probe.weights64_probe(rows.ctypes.data, got.ctypes.data, n)
    worst = F(0)
    for r, g in zip(rows, got):
        eps = F(12, 10 ** 6) * F(r[5]) ** 2 + F(floor12)
        u = [F(r[0]) + 2 * F(r[3]), F(r[3]) + F(r[4]), F(r[2]) - 2 * F(r[4])]
        s = [13 * F(r[k]) ** 2 + 3 * u[k] ** 2 + eps for k in range(3)]
        a, b, c = [1 / x ** 2 for x in s]
        left, right = a + 6 * b + 3 * c, 3 * a + 6 * b + c
        for have, want in zip(g, (2 * a / left, 3 * c / left, 3 * a / right, 2 * c / right)):
            worst = max(worst, abs(F(float(have)) - want) / want)
    assert worst <= F(1, 2 ** 51), float(worst)


def test_weights_are_finite_whatever_comes_in(probe):
    bad = [0.0, np.inf, -np.inf, np.nan, 5e-324, 1.7e308, -0.0]
    rng = np.random.default_rng(1)
    rows = rng.choice(bad, size=(2000, 7))
    rows[:, 5] = np.abs(rows[:, :5]).max(axis=1)  # as in a window: no difference is beyond its largest value's scale
    rows[:, 6] = 12e-99
    got = np.empty((len(rows), 4))
    probe.weights64_probe(rows.ctypes.data, got.ctypes.data, len(rows))
    assert np.isfinite(got).all() and (got >= 0).all() and (got <= 3.0).all()
