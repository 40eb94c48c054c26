"""Rotation groups with three real products a complex product, on the host: against the
same basis change with exact integers (each output sums 2, 4 or 8 rounded products; a
product drops at most 1/2 unit of 2^-60 of low limbs in the 32-bit form and 3/2 in the
pairs, and rounds by 1/2), and against the rotations themselves in exact rationals, for
every reflection pattern, for values at the norm bound and for axis-aligned angles."""
import ctypes
import math
import os
import subprocess
import tempfile
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def gc():
    so = os.path.join(tempfile.mkdtemp(), "gauss_check.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC",
                    "-I", os.path.join(ROOT, "paper_2212_14201_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "native", "gauss_check.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


def op(theta, reflect):
    c, s = math.cos(theta), math.sin(theta)
    return np.array([c, s, s, -c] if reflect else [c, -s, s, c])


def angles(rng, q, trial):
    if trial == 0:
        return [0.0] * q
    if trial == 1:
        return [math.pi / 2 * (k % 4) for k in range(q)]
    return list(rng.uniform(0, 2 * math.pi, q))


def values(rng, n, trial):
    v = rng.standard_normal(n)
    if trial % 3 == 1:
        v = np.sign(v)
    if trial % 3 == 2:
        v = np.zeros(n)
        v[rng.integers(n)] = 1.0
    v *= (1.25 if trial % 2 else 2.0 ** -14) / np.linalg.norm(v)
    return [int(round(float(t) * 2.0 ** 60)) for t in v]


def channels(z, coef, unit):
    """The basis change, the exact products and the inverse on z = [(re, im)]."""
    z = [list(t) for t in z]
    bits = [1 << b for b in range((len(z) - 1).bit_length())]
    for bit in bits:
        for j in range(len(z)):
            if not j & bit:
                lo, hi = z[j], z[j | bit]
                z[j], z[j | bit] = [lo[0] - hi[1], lo[1] + hi[0]], [lo[0] + hi[1], lo[1] - hi[0]]
    z = [[(c * a - d * b) / unit, (c * b + d * a) / unit] for (a, b), (c, d) in zip(z, coef)]
    for bit in reversed(bits):
        for j in range(len(z)):
            if not j & bit:
                A, B = z[j], z[j | bit]
                z[j], z[j | bit] = [A[0] + B[0], A[1] + B[1]], [A[1] - B[1], B[0] - A[0]]
    return z


def rotate(x, ops):
    x = [Fraction(v) for v in x]
    for q, m in enumerate(ops):
        m = [Fraction(float(t)) for t in m]
        for j in range(len(x)):
            if not j >> q & 1:
                a, b = x[j], x[j | 1 << q]
                x[j], x[j | 1 << q] = m[0] * a + m[1] * b, m[2] * a + m[3] * b
    return x


@pytest.mark.parametrize("q", [2, 3, 4])
def test_group(gc, q):
    fn = {2: gc.gc_pair, 3: gc.gc_triple, 4: gc.gc_quad}[q]
    rng = np.random.default_rng(70 + q)
    per_product = Fraction(2) if q == 2 else Fraction(1)
    for flags in range(1 << q):
        for trial in range(14):
            th = angles(rng, q, trial)
            ops = [op(th[k], flags >> k & 1) for k in range(q)]
            x = values(rng, 1 << q, trial)
            buf = (ctypes.c_longlong * (1 << q))(*x)
            cf = (ctypes.c_longlong * (1 << q))()
            ptrs = [o.ctypes.data_as(ctypes.c_void_p) for o in ops]
            assert fn(*ptrs, buf, cf) == flags
            got = list(buf)
            fx = [-v if bin(k & flags).count("1") & 1 else v for k, v in enumerate(x)]
            # pairs along the first bit; channels over the other bits.  A triple orders its
            # channels by the reversed bits (U+, U-, V+, V-)
            n = 1 << (q - 1)
            order = [0, 2, 1, 3] if q == 3 else list(range(n))
            coef = [None] * n
            for k in range(n):
                coef[order[k]] = (cf[2 * k], cf[2 * k + 1])
            unit = Fraction(2) ** (60 if q == 2 else 64)
            z = channels([(Fraction(fx[2 * j]), Fraction(fx[2 * j + 1])) for j in range(n)], coef, unit)
            want = [t for pair in z for t in pair]
            assert max(abs(a - b) for a, b in zip(got, want)) <= n * per_product
            # the rotations themselves: coefficients carry double rounding (their angles'
            # cosines and products, a few 2^-53 of the value) besides the bound above
            exact = rotate(x, ops)
            size = Fraction(math.isqrt(sum(v * v for v in x)) + 1)
            assert max(abs(a - b) for a, b in zip(got, exact)) <= n * per_product + size * Fraction(24, 2 ** 53)
