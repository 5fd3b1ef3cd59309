"""CPU check of the FP32 rounding that the updates of FP32 blocks use where the
lean form declines (fx.cuh, compiled here for the host through a small shim):
one rounding of the exact sum, against exact rational arithmetic."""
import ctypes as C
import os
import random
import shutil
import struct
import subprocess
from fractions import Fraction as F

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1806_01036_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("flt") / "libflt.so")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", CSRC,
                    os.path.join(ROOT, "tests", "fxshim", "float_shim.cu"), "-o", out], check=True, capture_output=True)
    L = C.CDLL(out)
    L.flt_w_to_float.argtypes = [C.c_longlong, C.c_longlong, C.c_int]
    L.flt_w_to_float.restype = C.c_float
    return L


def nearest(x):
    """Bits of the FP32 nearest to the rational x (ties to even)."""
    sign, x = (0x80000000, -x) if x < 0 else (0, x)
    if x == 0:
        return 0
    e = max(x.numerator.bit_length() - x.denominator.bit_length() - 1, -126)
    if x >= F(2) ** (e + 1):
        e += 1
    e = max(e, -126)
    q = x / F(2) ** (e - 23)
    m = q.numerator // q.denominator
    rest = q - m
    if rest > F(1, 2) or (rest == F(1, 2) and m & 1):
        m += 1
    if m >> 24:
        m, e = m >> 1, e + 1
    if e > 127:
        return sign | 0x7f800000
    return sign | (m if not m >> 23 else ((e + 127) << 23) | (m & 0x7fffff))


def bits(f):
    return struct.unpack("<I", struct.pack("<f", f))[0]


def test_sums_are_rounded_once(lib):
    g = random.Random(5)
    for i in range(20000):
        n = g.randint(1, 126)
        w = g.getrandbits(n)
        kind = i % 5
        if kind == 1:  # a tie of 24 bits, or one unit to either side of it, far below
            n = g.randint(60, 120)
            w = ((g.getrandbits(24) | 1 << 23) << 1 | 1) << (n - 25)
            w += g.choice([-1, 0, 1])
        elif kind == 2:  # the same beside a representable value
            n = g.randint(60, 120)
            w = ((g.getrandbits(24) | 1 << 23) << (n - 24)) + g.choice([-1, 0, 1])
        w *= g.choice([-1, 1])
        S = g.randint(-200, 20) - (abs(w).bit_length() if kind == 3 else 0)
        if kind == 4:  # near the largest and the smallest FP32 numbers
            S = g.choice([127, 128, -126, -149, -150]) - abs(w).bit_length() + g.randint(-1, 2)
        v = w & (1 << 128) - 1
        got = lib.flt_w_to_float(C.c_longlong(v & 2 ** 64 - 1).value, C.c_longlong(v >> 64).value, S)
        want = nearest(F(w) * F(2) ** S)
        assert bits(got) == (want | (0x80000000 if w < 0 else 0)), (w, S)
