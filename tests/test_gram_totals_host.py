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


def rows():
    g = random.Random(7)
    edges = [1 << b for b in range(27)]
    return sorted({r + d for r in edges for d in (-1, 0, 1) if r + d >= 1} | {g.randrange(1, 1 << 26) for _ in range(500)})


def test_totals_hold_the_sum_of_their_rows(lib):
    """The largest values that an alignment exponent allows are below 2^110
    units, so a product is below 2^124 of the sums' units (2^220 / 2^96, the kept
    digit pairs a little more).  Their sum over the rows, less the dropped bits,
    fits a signed 128-bit total; the rows are those of all parts of a chunk, up
    to 16 x 2^22."""
    for r in rows():
        drop = lib.tots_fold_bits(r)
        assert r * (2 ** 124 + 2 ** 110) >> drop < 2 ** 127
        assert drop >= 0


@pytest.mark.parametrize("lanes,spacing,most", [(24, 90_000, 1 << 26), (8, 13_000, 1 << 22)])
def test_dropped_bits_cost_less_than_the_dropped_pairs(lib, lanes, spacing, most):
    """A fold rounds a lane down by less than 2^drop units of the sums; an entry of
    a symmetric tile adds 24 lanes, folded every 90,000 rows of a part or less
    often (960 rows a drain, 96 drains), one of X^T Y at most 8, every 13,000.
    max|x| max|y| is at least 2^214 / 2^96 = 2^118 of these units, so a product's
    share stays below 2^-108 of it."""
    for r in rows():
        if r <= most:
            folds = 1 + r // spacing // (16 if r > 1 << 22 else 1)
            assert F(lanes * folds * 2 ** lib.tots_fold_bits(r), r) / 2 ** 118 <= F(2) ** -108, r
