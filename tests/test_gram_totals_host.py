"""CPU checks of the integer totals of the tensor-core Gram products (fx.cuh,
compiled here for the host through a small shim) against Python's integers."""
import ctypes as C
import os
import random
import shutil
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
    out = str(tmp_path_factory.mktemp("tot") / "libtot.so")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", CSRC,
                    os.path.join(ROOT, "tests", "fxshim", "total_shim.cu"), "-o", out], check=True, capture_output=True)
    return C.CDLL(out)


def words(v):
    v &= (1 << 128) - 1
    return [C.c_longlong(v & (2 ** 64 - 1)).value, C.c_longlong(v >> 64).value]


def signed(lo, hi):
    return (hi << 64) | (lo & (2 ** 64 - 1))


@pytest.mark.parametrize("spare", [1, 2, 3, 4])
def test_sum_of_parts(lib, spare):
    """2^spare parts of any size up to the 127 bits a part may take, each with a
    scale of its own: the sum is off by less than one unit of its scale for
    every part and shift, and that unit is below 2^-(126 - spare) of the largest part or
    a unit of the parts' largest scale."""
    g = random.Random(7)
    m = 1 << spare
    for trial in range(2000):
        top = 1 if trial % 4 else 0
        v, s = [], []
        for i in range(m):
            bits = 127 if not top else g.choice([0, 1, 60, 100, 120, 124, 126, 127])
            x = (1 << bits) - 1 if trial % 2 else g.getrandbits(bits) if bits else 0
            v.append(-x - 1 if g.random() < 0.4 and trial % 8 else x)
            s.append(-2000 + (0 if trial % 3 else g.randrange(0, 12)))
        w = (C.c_longlong * (2 * m))(*[t for x in v for t in words(x)])
        out, so = (C.c_longlong * 2)(), C.c_int()
        lib.tots_sum(spare, w, (C.c_int * m)(*s), out, C.byref(so))
        got = F(signed(out[0], out[1])) * F(2) ** so.value
        want = sum(F(x) * F(2) ** e for x, e in zip(v, s))
        unit = F(2) ** so.value
        assert abs(got - want) <= 2 * m * unit
        assert so.value <= max(s) + spare
        assert so.value == max(s) or max(abs(F(x)) * F(2) ** e for x, e in zip(v, s)) >= 2 ** (126 - spare) * unit / 2 ** spare


@pytest.mark.parametrize("spare", [0, 1, 4])
def test_totals_keep_their_low_bits(lib, spare):
    """The sum of terms w + lo 2^-20 is exact, its shift rounds down by less than
    2^-20, and narrowing it drops only what 127 - spare bits cannot hold."""
    g = random.Random(11)
    for trial in range(3000):
        m = g.randint(1, 6)
        bits = g.choice([0, 1, 40, 90, 106, 107, 110, 123])
        v = [g.getrandbits(bits) * g.choice([-1, 1]) if bits else 0 for _ in range(m)]
        lo = [g.getrandbits(20) if trial % 3 else g.choice([0, (1 << 20) - 1]) for _ in range(m)]
        sh = g.choice([0, 0, 1, 7, 19, 20, 21, 60, 126, 127, 300])
        out, so = (C.c_longlong * 2)(), C.c_int()
        lib.tots_total(m, (C.c_longlong * (2 * m))(*[t for x in v for t in words(x)]), (C.c_uint * m)(*lo), sh, spare,
                       out, C.byref(so))
        got = signed(out[0], out[1])
        full = sum((x << 20) + l for x, l in zip(v, lo))  # units 2^-20
        full = full >> sh if sh < 127 else 0
        assert abs(got) <= 1 << (127 - spare)
        assert -20 <= so.value <= spare
        assert got == full >> (so.value + 20)
        if so.value > -20:
            assert abs(got) >= 1 << (126 - spare - 1)
