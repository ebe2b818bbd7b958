"""The FP64 polynomials and tables: the committed poly64.cuh is its generator's output, and
the FP64 tanh and reciprocal square root built on them (emulated in numpy, with FP32 seeds of
the hardware's accuracy) are within a few units in the last place of mpmath."""
import os
import re
import subprocess
import sys

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_01234_gb300", "csrc")
SRC = open(os.path.join(CSRC, "poly64.cuh")).read()
EPS = 2.0 ** -52


def fma(a, b, c):
    """One rounding in extended precision, one to FP64."""
    return (np.longdouble(a) * np.longdouble(b) + np.longdouble(c)).astype(np.float64)


def table(name):
    return np.array([float(v) for v in re.search(name + r"\[32\] = \{([^}]*)\}", SRC).group(1).split(",") if v.strip()])


def constant(name):
    return float(re.search(name + r" = ([^,;]+)[,;]", SRC).group(1))


def test_committed_file_is_generated():
    out = subprocess.run([sys.executable, os.path.join(CSRC, "gen_poly64.py")], capture_output=True, text=True)
    assert out.returncode == 0, out.stderr
    assert out.stdout == SRC


def test_tanh():
    rng = np.random.default_rng(1)
    x = np.concatenate([rng.uniform(-19.99, 19.99, 2000), rng.uniform(-1, 1, 2000), 10.0 ** rng.uniform(-12, 0, 500)])
    t = -2.0 * np.abs(x)
    s = fma(t, constant("kLn2Inv"), 6755399441055744.0)
    nd = s - 6755399441055744.0
    n = nd.astype(np.int64)
    r = fma(-nd, constant("kLn2Lo"), fma(-nd, constant("kLn2Hi"), t))
    p = fma(r, 1 / 720, 1 / 120)
    for c in (1 / 24, 1 / 6, 0.5):
        p = fma(p, r, c)
    p = fma(p * r, r, r)
    em = np.ldexp(table("kExp2Table")[n & 31], n >> 5)
    m = fma(em, p + table("kExp2Rest")[n & 31], em - 1.0)
    d = 2.0 + m
    y = (np.float32(1) / d.astype(np.float32) * np.float32(1 + 2.0 ** -22)).astype(np.float64)  # a seed 2 ulp off
    e = fma(-d, y, 1.0)
    h = np.copysign(-m * fma(y, fma(e, e, e), y), x)
    want = np.array([float(mp.tanh(mp.mpf(float(v)))) for v in x])
    assert np.max(np.abs(h - want) / np.abs(want)) < 4 * EPS


def test_rsqrt():
    v = 10.0 ** np.random.default_rng(2).uniform(-6, 6, 4000)
    y = (1 / np.sqrt(v.astype(np.float32)) * np.float32(1 + 2.0 ** -22)).astype(np.float64)
    e = fma(-(v * y), y, 1.0)
    z = fma(y * e, fma(0.375, e, 0.5), y)
    want = np.array([float(1 / mp.sqrt(mp.mpf(float(q)))) for q in v])
    assert np.max(np.abs(z - want) / want) < 2 * EPS
