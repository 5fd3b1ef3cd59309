"""CPU checks of the 128-bit floating point that the k-by-k steps of the
compensated modes run (paper_1806_01036_gb300/csrc/wide.cuh, compiled here for
the host through a small shim) against exact rational arithmetic."""
import ctypes as C
import math
import os
import random
import shutil
import subprocess
from fractions import Fraction as F

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1806_01036_gb300", "csrc")
ADD, SUB, MUL, DOT2, RECIP, RSQRT, SQRT = range(7)
A4 = C.c_ulonglong * 4


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("wide") / "libwide.so")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", CSRC,
                    os.path.join(ROOT, "tests", "fxshim", "wide_shim.cu"), "-o", out], check=True, capture_output=True)
    L = C.CDLL(out)
    L.wides_from.argtypes = [C.c_double, C.c_double, A4]
    L.wides_to.argtypes = [A4, C.POINTER(C.c_double), C.POINTER(C.c_double)]
    return L


def value(w):
    m = (w[0] << 64) | w[1]
    assert m == 0 or m >> 127, "not normalized"
    e = C.c_longlong(w[2]).value
    v = F(m) * F(2) ** (e - 127) if m else F(0)
    return -v if w[3] else v


def make(m, e, s):
    return A4(m >> 64, m & (2 ** 64 - 1), C.c_ulonglong(e & (2 ** 64 - 1)).value, s)


ZERO = (0, -(1 << 28), 0)


def rand(g, spread=40):
    kind = g.randrange(6)
    if kind == 0:
        m = 1 << 127
    elif kind == 1:
        m = (1 << 128) - 1
    elif kind == 2:
        m = (1 << 127) | g.getrandbits(20)
    elif kind == 3:
        m = g.getrandbits(53) << 75 | 1 << 127
    else:
        m = g.getrandbits(127) | 1 << 127
    return make(m, g.randint(-spread, spread), g.randrange(2))


def run(L, op, a, b=None, c=None, d=None):
    r = A4()
    L.wides_op(op, a, b or a, c or a, d or a, r)
    return r


def test_sums_and_products(lib):
    g = random.Random(1)
    for i in range(6000):
        spread = (2, 40, 150)[i % 3]
        a, b, c, d = (rand(g, spread) for _ in range(4))
        if i % 7 == 0:
            b = make((a[0] << 64 | a[1]) ^ g.getrandbits(3) or 1 << 127, C.c_longlong(a[2]).value, a[3])
            if not (b[0] >> 63):
                b = a
        if i % 50 == 0:
            b = make(*ZERO)
        x, y, z, w = map(value, (a, b, c, d))
        for op, ref in ((ADD, x + y), (SUB, x - y)):
            assert abs(value(run(lib, op, a, b)) - ref) <= F(2) ** -124 * max(abs(x), abs(y)), (op, i)
        assert abs(value(run(lib, MUL, a, b)) - x * y) <= F(2) ** -124 * abs(x * y)
        got = value(run(lib, DOT2, a, b, c, d))
        assert abs(got - (x * y + z * w)) <= F(2) ** -122 * max(abs(x * y), abs(z * w)), i


def test_exact_cases(lib):
    g = random.Random(2)
    for _ in range(1000):
        p, q = g.randint(1, 2 ** 60), g.randint(1, 2 ** 60)
        a, b = A4(), A4()
        hi = float(p)
        lib.wides_from(hi, float(p - int(hi)), a)
        hi = float(q)
        lib.wides_from(hi, float(q - int(hi)), b)
        assert value(a) == p and value(b) == q
        assert value(run(lib, ADD, a, b)) == p + q
        assert value(run(lib, SUB, a, b)) == p - q
        assert value(run(lib, MUL, a, b)) == p * q
    for e in range(-7, 8):
        a = make(1 << 127, 2 * e, 0)
        assert value(run(lib, RSQRT, a)) == F(2) ** -e
        assert value(run(lib, SQRT, a)) == F(2) ** e
        assert value(run(lib, RECIP, a)) == F(2) ** (-2 * e)


def test_reciprocals_and_roots(lib):
    g = random.Random(3)
    for i in range(4000):
        a = rand(g, 300)
        x = value(a)
        assert abs(value(run(lib, RECIP, a)) * x - 1) <= F(2) ** -116
        a = make(a[0] << 64 | a[1], C.c_longlong(a[2]).value, 0)
        x = abs(x)
        y = value(run(lib, RSQRT, a))
        assert abs(y * y * x - 1) <= F(2) ** -116, i
        s = value(run(lib, SQRT, a))
        assert abs(s * s / x - 1) <= F(2) ** -115


def test_conversions(lib):
    g = random.Random(4)
    for i in range(4000):
        hi = g.choice([-1, 1]) * math.ldexp(1 + g.random(), g.randint(-1000, 1000))
        if i % 20 == 0:
            hi = g.choice([0.0, -0.0, 5e-324, -1e-310, 1.0])
        lo = math.ulp(hi) * g.uniform(-0.5, 0.5) if abs(hi) > 1e-290 else 0.0
        hi, lo = hi + lo, lo - ((hi + lo) - hi)
        a = A4()
        lib.wides_from(hi, lo, a)
        x = F(hi) + F(lo)
        assert abs(value(a) - x) <= F(2) ** -124 * abs(x)
        h, l = C.c_double(), C.c_double()
        lib.wides_to(a, h, l)
        assert h.value == hi
        assert abs(F(h.value) + F(l.value) - x) <= F(2) ** -106 * abs(x) + F(2) ** -1074
