"""The tensor-core row engine at the edges of its tiles: K widths 16, 32 and 64
on either side, one and two output blocks, row counts on either side of a tile
and of one and two tiles a CTA, and tiles that need all fourteen digits
(values on either side of the near window, 25 binades below the row's largest,
subnormals, rows of widely different scale) among tiles that need ten, in
several orders.

Bound: every product is off by less than kv 2^-99 of the row's and the column's
largest values (the engine's own bound, 2^-103 per product, lies below it); the
sum is exact and rounded once."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a.T)).cuda().t()


def check(eo, ctx, monkeypatch, v, k, seed):
    import torch

    monkeypatch.setenv("EO_DD_ROW_ENGINE", "umma")
    n, kv = v.shape
    g = synth.rng(seed)
    y = synth.gaussian(n, k, seed + 1) * 1e-3
    ch = np.asfortranarray(g.standard_normal((kv, k)))
    cl = np.asfortranarray(ch * 2.0 ** -55 * g.uniform(-1, 1, (kv, k)))
    out, _ = eo.project_apply(ctx, dev(v), dev(y), (dev(ch), dev(cl)), prec=eo.DD, want_m=False)
    ref = oracle.project_apply(v, y, ch, cl)
    row_max = np.max(np.abs(v), axis=1)[:, None] * np.max(np.abs(ch) + np.abs(cl), axis=0)[None, :]
    err = np.abs(out.cpu().numpy() - ref)
    assert np.all(err <= 2 * U * np.abs(ref) + kv * 2.0 ** -99 * row_max + 5e-324)


@pytest.mark.parametrize("kv,k", [(15, 16), (16, 4), (17, 16), (31, 17), (32, 32), (33, 16), (63, 5), (64, 16)])
@pytest.mark.parametrize("n", [1, 128, 129, 152 * 128 - 1, 152 * 128 + 1, 304 * 128 + 130])
def test_tile_edges(eo, ctx, monkeypatch, n, kv, k):
    check(eo, ctx, monkeypatch, synth.gaussian(n, kv, 2000 + kv + n % 89), k, 2100 + k)


@pytest.mark.parametrize("kv,k", [(16, 16), (12, 3), (32, 16), (20, 8), (32, 32), (20, 17), (64, 16), (40, 9)])
@pytest.mark.parametrize("kind", ["some", "alternate", "all", "window", "zeros"])
def test_tiles_of_both_kinds(eo, ctx, monkeypatch, kind, kv, k):
    n = 152 * 128 * 4 + 77
    g = synth.rng(2200 + kv + k)
    v = synth.gaussian(n, kv, 2300 + kv)
    tile = np.arange(n) // 128
    if kind == "some":  # single values far below their row, here and there
        r, c = g.integers(0, n, 60), g.integers(0, kv, 60)
        v[r, c] *= 2.0 ** -g.integers(18, 140, 60).astype(float)
        v[g.integers(0, n, 6), g.integers(0, kv, 6)] = 5e-324
    elif kind == "alternate":  # every other of a CTA's tiles
        v[(tile // 152) % 2 == 1, 0] *= 2.0 ** -60
        v *= np.ldexp(1.0, g.integers(-200, 200, n))[:, None]
    elif kind == "all":
        v *= np.ldexp(1.0, g.integers(-120, 1, (n, kv)))
    elif kind == "window":  # binades 23 to 27 below the row's largest
        v = np.where(g.random((n, kv)) < 0.5, -1.0, 1.0) * (1 + g.random((n, kv)))
        v *= np.ldexp(1.0, -g.integers(23, 28, (n, kv)) * (np.arange(kv) > 0))
        v[tile % 3 == 0, 1:] *= 4.0
    else:
        v[g.random((n, kv)) < 0.01] = 0.0
        v[g.integers(0, n, 40)] = 0.0
        v[g.integers(0, n, 40), 0] = -0.0
    check(eo, ctx, monkeypatch, np.asfortranarray(v), k, 2400 + k)


@pytest.mark.parametrize("n,k", [(16384, 9), (16383, 16), (20_011, 16), (20_011, 17), (152 * 128 + 1, 32), (20_000, 8),
                                 (20_000, 33)])
@pytest.mark.parametrize("spread", [0, 60])
def test_f32_update(eo, ctx, n, k, spread):
    """Q = X R^-1 of an FP32 block, on either side of the digit engine's sizes,
    rows of widely different scale and a column far below the others (tiles
    that need all digits) included.  Q is one FP32 rounding (2^-24 relative;
    2^-23 allows for R^-1 formed here in FP64) of X R^-1, whose error is k 2^-48
    of the row's and the column's largest values at most."""
    import torch

    g = synth.rng(2500 + k)
    x = g.standard_normal((n, k))
    if spread:
        x *= np.ldexp(1.0, g.integers(-spread // 2, 1, n))[:, None]
        x[:, k // 2] *= 2.0 ** -spread
    x = x.astype(np.float32)
    X = torch.from_numpy(np.ascontiguousarray(x.T)).cuda().t()
    rh, rl, info = eo.cholqr(ctx, X, passes=1, prec=eo.F32)
    assert int(info) == 0
    z = np.linalg.inv((rh + rl).cpu().numpy())
    want = x.astype(np.float64) @ z
    err = np.abs(X.cpu().numpy().astype(np.float64) - want)
    row_max = np.max(np.abs(x), axis=1)[:, None].astype(np.float64) * np.max(np.abs(z), axis=0)[None, :]
    assert np.all(err <= 2.0 ** -23 * np.abs(want) + k * 2.0 ** -48 * row_max)
