"""CPU check of the row kernels' word-wise roundings (w_to_double_lean and
sub_round_lean of fx.cuh) against the general ones: the same bits wherever they
report ok, and ok wherever the result is a normal double whose bits below the
rounding are neither nearly all zeros nor nearly all ones."""
import ctypes as C

import numpy as np

from test_fx_host import F, _bits, fx, split_w  # noqa: F401  (fx is a fixture)

OFFSET = sum(0x8B400000 << (16 * m) for m in range(7)) % (1 << 128)


def plain(q):
    """The 43 bits of |q| below its 53 leading ones lie off 0 and off 2^43 by more than 2^12."""
    q = abs(q)
    if q == 0:
        return False
    n, d = q.numerator, q.denominator
    e = n.bit_length() - d.bit_length()
    sh = 96 - e
    v = (n << sh) // d if sh >= 0 else n // (d << -sh)
    while v >= 1 << 96:
        v >>= 1
    low = v % (1 << 32)
    return 1 << 12 < low < (1 << 32) - (1 << 12)


def rand_w(g):
    bits = int(g.integers(1, 123))
    w = int(g.integers(0, 2 ** 62)) << 62 | int(g.integers(0, 2 ** 62))
    w %= 1 << bits
    kind = g.random()
    if kind < 0.15 and bits > 60:  # a tie or an exact double
        w = (w >> (bits - 53) << (bits - 53)) | (int(g.integers(0, 2)) << (bits - 54))
    elif kind < 0.3:  # runs of zeros or ones at the end
        t = int(g.integers(1, bits + 1))
        w = (w >> t << t) | (((1 << t) - 1) if g.random() < 0.5 else 0)
    if g.random() < 0.2:
        w += int(g.integers(-3, 4))
    return -w if g.random() < 0.5 else w


def test_lean_product_rounding(fx):
    fx.fxs_w_to_double_lean.restype = C.c_double
    fx.fxs_w_to_double_lean.argtypes = [C.c_longlong, C.c_longlong, C.c_int, C.c_int, C.c_void_p]
    g = np.random.default_rng(31)
    ok = C.c_int(0)
    must = 0
    for _ in range(20000):
        w = rand_w(g)
        S = int(g.integers(-1300, 1000)) if g.random() < 0.15 else int(g.integers(-300, 100))
        flip = int(g.integers(0, 2))
        got = fx.fxs_w_to_double_lean(*split_w(w), S, flip, C.byref(ok))
        want = fx.fxs_w_to_double(*split_w(w), S)
        if ok.value:
            assert _bits(got) == _bits(-want if flip else want), (w, S)
        if abs(w) >= 2 ** 64 and 2.0 ** -1021 <= abs(want) < 2.0 ** 1022 and plain(F(w)):
            must += 1
            assert ok.value, (w, S)
    assert must > 4000


def test_lean_difference_rounding(fx):
    ll = C.c_longlong
    fx.fxs_sub_round_lean.restype = C.c_double
    fx.fxs_sub_round_lean.argtypes = [C.c_double, ll, ll, ll, ll, C.c_int, C.c_void_p]
    g = np.random.default_rng(32)
    ok = C.c_int(0)
    must = 0
    for _ in range(30000):
        y = float(np.ldexp(g.standard_normal(), int(g.integers(-80, 80))))
        S = int(g.integers(-300, -30))
        mode = int(g.integers(0, 4))
        if mode == 0:  # cancellation
            w = int(F(y) / F(2) ** S) + int(g.integers(-10 ** 6, 10 ** 6)) * 2 ** int(g.integers(0, 80))
        elif mode == 1:  # y dominating by 0 .. 260 binades
            e = int(np.frexp(abs(y))[1]) - int(g.integers(0, 260))
            w = rand_w(g)
            S = e - abs(w).bit_length()
        else:
            w = rand_w(g)
            if g.random() < 0.8:  # y's last bit -20 .. 140 places above the grid
                S = int(np.frexp(abs(y))[1]) - 53 - int(g.integers(-20, 140))
        if g.random() < 0.02:
            y = [0.0, -0.0, 5e-324, float("inf")][int(g.integers(0, 4))]
        if not -(1 << 122) < w < (1 << 122):
            continue
        K = OFFSET if g.random() < 0.8 else 0
        got = fx.fxs_sub_round_lean(y, *split_w(w), *split_w(K), S, C.byref(ok))
        normal = np.isfinite(y) and abs(y) >= 2.0 ** -1022
        if ok.value:
            assert normal
            assert _bits(got) == _bits(fx.fxs_sub_round(y, *split_w(w), S)), (y, w, S)
        if normal:
            exact = F(y) - F(w) * F(2) ** S
            d = int(np.frexp(abs(y))[1]) - 53 - S
            if d >= 0 and 2.0 ** -1000 < abs(exact) < 2 ** 1000 and plain(exact) and abs(exact) >= F(2) ** (S + 64) and d < 72:
                must += 1
                assert ok.value, (y, w, S)
    assert must > 3000


def test_lean_single_rounding_and_widening(fx):
    fx.fxs_w_to_float_lean.restype = C.c_float
    fx.fxs_w_to_float_lean.argtypes = [C.c_longlong, C.c_longlong, C.c_int, C.c_void_p]
    fx.fxs_widen.restype = C.c_double
    fx.fxs_widen.argtypes = [C.c_float]
    g = np.random.default_rng(33)
    ok = C.c_int(0)
    must = 0
    for _ in range(20000):
        w = rand_w(g)
        S = int(g.integers(-240, 120))
        got = np.float32(fx.fxs_w_to_float_lean(*split_w(w), S, C.byref(ok)))
        exact = F(w) * F(2) ** S
        if ok.value:
            assert 2.0 ** -126 <= abs(got) < np.inf
            err = abs(F(float(got)) - exact)
            for side in (np.float32(np.inf), np.float32(-np.inf)):
                other = np.nextafter(got, side)
                if np.isfinite(other):
                    assert err <= abs(F(float(other)) - exact), (w, S)
        v = abs(w) << 128 >> max(abs(w).bit_length() + 128 - 64, 0)  # the 64 leading bits
        if abs(w) >= 2 ** 64 and F(2) ** -125 <= abs(exact) < F(2) ** 126 and 1 << 12 < v % 2 ** 32 < 2 ** 32 - (1 << 12):
            must += 1
            assert ok.value, (w, S)
    assert must > 4000
    for x in (0.0, -0.0, 1.0, -1.5, 1e-45, -1e-40, 1.17549435e-38, 3.4028235e38, float("inf"), -float("inf")):
        assert _bits(fx.fxs_widen(x)) == _bits(float(np.float32(x)))
    assert np.isnan(fx.fxs_widen(float("nan")))
    for x in g.standard_normal(500).astype(np.float32) * np.float32(2.0) ** g.integers(-60, 60, 500).astype(np.float32):
        assert fx.fxs_widen(float(x)) == float(x)
