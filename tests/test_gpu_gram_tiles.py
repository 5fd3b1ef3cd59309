"""The tensor-core Gram engine at the edges of its tiles: column counts on
either side of its 8-, 16-, 32- and 64-column tiles and of the narrow products
that the integer limbs keep, row counts on either side
of a K step, of a panel and of a row chunk, TMA and element-wise loads, and
values on either side of the near window (25 binades below the alignment
exponent), zeros and growing exponents among them.

Bound: every product is off by less than 2^-96 max|x_i| max|y_j| (the engine's
own bound, 2^-103, lies below it), the sums are exact and the result is rounded
once to a double-double: |G - G*| <= 2^-104 |G*| + n 2^-96 max|x_i| max|y_j|."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def check(eo, ctx, x, y, odd_ld=False):
    import torch

    def dev(a):
        n, k = a.shape
        ld = n + 1 - n % 2 if odd_ld else n + n % 2  # an even leading dimension: TMA
        t = torch.full((k, ld), float("nan"), dtype=torch.float64, device="cuda")
        t[:, :n] = torch.from_numpy(np.ascontiguousarray(a.T))
        return t.t()[:n]

    gh, gl = eo.gram(ctx, dev(x), None if y is x else dev(y))
    rh, rl = oracle.gram(x, None if y is x else y)
    err = np.abs((gh.cpu().numpy() - rh) + (gl.cpu().numpy() - rl))
    tol = 2.0 ** -104 * np.abs(rh) + x.shape[0] * 2.0 ** -96 * np.outer(np.abs(x).max(0), np.abs(y).max(0))
    assert np.all(err <= tol), float(np.max(err / np.where(tol > 0, tol, 1)))


@pytest.mark.parametrize("odd_ld", [False, True])
@pytest.mark.parametrize("kx,ky", [(9, 1), (16, 8), (17, 9), (32, 16), (33, 8), (64, 17), (3, 40), (16, 0), (17, 0), (64, 0),
                                   (4, 0), (5, 0), (8, 0), (8, 3), (8, 4), (5, 7)])
def test_column_tiles(eo, ctx, kx, ky, odd_ld):
    x = synth.gaussian(12_345, kx, 900 + kx)
    check(eo, ctx, x, synth.gaussian(12_345, ky, 950 + ky) if ky else x, odd_ld)


@pytest.mark.parametrize("n", [1, 15, 16, 17, 47, 48, 49, 63, 65, 239, 241, 152 * 64 - 1, 152 * 64 + 1, 152 * 240 + 1])
@pytest.mark.parametrize("kx,ky", [(64, 16), (16, 0)])
def test_row_edges(eo, ctx, n, kx, ky):
    x = synth.gaussian(n, kx, 1000 + n % 97)
    check(eo, ctx, x, synth.gaussian(n, ky, 1100 + n % 97) if ky else x)


@pytest.mark.parametrize("kind", ["zeros", "below", "grow", "zero column", "mixed"])
@pytest.mark.parametrize("kx,ky", [(20, 12), (64, 16), (30, 5), (16, 0), (10, 0), (12, 9), (5, 0), (8, 8)])
@pytest.mark.parametrize("odd_ld", [False, True])
def test_special_panels(eo, ctx, kind, kx, ky, odd_ld):
    n = 30_011
    g = synth.rng(1200 + kx + ky)
    x = synth.gaussian(n, kx, 1300 + kx)
    y = synth.gaussian(n, ky, 1400 + ky) if ky else x
    for a in (x, y) if ky else (x,):
        k = a.shape[1]
        if kind in ("zeros", "mixed"):
            a[g.random(a.shape) < 1e-3] = 0.0
            a[g.integers(0, n, 20), g.integers(0, k, 20)] = -0.0
        if kind in ("below", "mixed"):
            r, c = g.integers(0, n, 40), g.integers(0, k, 40)
            a[r, c] *= 2.0 ** -g.integers(18, 140, 40).astype(float)
            a[g.integers(0, n, 4), g.integers(0, k, 4)] = 5e-324
        if kind in ("grow", "mixed"):
            for i in range(6):
                a[g.integers(0, n), g.integers(0, k)] *= 2.0 ** (7 * (i + 1))
        if kind == "zero column":
            a[:, k - 1] = 0.0
    check(eo, ctx, x, y, odd_ld)


@pytest.mark.parametrize("kind", ["plain", "mixed"])
@pytest.mark.parametrize("n", [256, 4096, 4097, 300_000, 300_255, 152 * 240 * 16])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 7, 8])
@pytest.mark.parametrize("odd_ld", [False, True])
def test_rows_in_parts(eo, ctx, monkeypatch, kind, n, k, odd_ld):
    """Symmetric products of up to 8 columns on the tensor cores: the rows in
    parts side by side, with and without rows left over, chunks of one panel and
    of several."""
    monkeypatch.setenv("EO_DD_GRAM_ENGINE", "umma")
    g = synth.rng(1500 + k + n % 97)
    x = synth.gaussian(n, k, 1600 + k)
    if kind == "mixed":
        x[n // 3:] *= 2.0 ** -9  # the parts' exponents differ
        x[g.random(x.shape) < 1e-3] = 0.0
        r, c = g.integers(0, n, 40), g.integers(0, k, 40)
        x[r, c] *= 2.0 ** -g.integers(18, 140, 40).astype(float)
        x[g.integers(0, n, 4), g.integers(0, k, 4)] = 5e-324
        for i in range(4):
            x[g.integers(0, n), g.integers(0, k)] *= 2.0 ** (7 * (i + 1))
    check(eo, ctx, x, x, odd_ld)


def test_rows_in_parts_non_finite(eo, ctx, monkeypatch):
    import torch

    monkeypatch.setenv("EO_DD_GRAM_ENGINE", "umma")
    for row in (0, 4095, 2500):
        x = synth.gaussian(4096, 4, 1700)
        x[row, 2] = np.inf if row else np.nan
        gh, _ = eo.gram(ctx, torch.from_numpy(np.ascontiguousarray(x.T)).cuda().t())
        assert bool(torch.isnan(gh[2, 2]))
