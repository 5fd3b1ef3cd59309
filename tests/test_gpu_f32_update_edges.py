"""FP32 updates X Z where the tensor-core digits meet their limits: values that
are not finite, and rows and columns of widely different scale."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(np.asarray(a).T)).cuda().t()


def fp64_update(x, z, tri):
    """x z row by row, as a chain of FP64 products and sums over the entries that
    the sum takes (i <= j of a triangular z)."""
    out = np.zeros(x.shape)
    with np.errstate(all="ignore"):
        for j in range(z.shape[1]):
            for i in range(j + 1 if tri else z.shape[0]):
                out[:, j] += x[:, i].astype(np.float64) * z[i, j]
        return out


@pytest.mark.parametrize("n,k", [(16_384, 9), (20_011, 16), (20_011, 17), (152 * 128 * 2 + 5, 32)])
def test_non_finite_values(eo, ctx, n, k):
    """With M given (the block's own, before the values were put in): an Inf or NaN
    in column i leaves the columns before i of its row alone, and makes the others
    what FP64 sums make of them.  Finite outputs: one FP32 rounding (2^-24, and
    2^-48 of the products for Z, which is formed here in FP64)."""
    x = synth.gaussian(n, k, 6500 + k).astype(np.float32)
    m = eo.gram(ctx, dev(x), prec=eo.F32)
    d = dev(x)
    rh, _, info = eo.cholqr(ctx, d, passes=1, prec=eo.F32, M=m)
    assert int(info) == 0
    z = np.linalg.inv(rh.cpu().numpy())
    g = synth.rng(6600 + k)
    rows = g.permutation(n)[:40]
    for r in rows[:30]:
        x[r, g.integers(0, k)] = g.choice([np.inf, -np.inf, np.nan])
    for r in rows[20:40]:
        x[r, g.integers(0, k)] = g.choice([np.inf, -np.inf])
    d = dev(x)
    _, _, info = eo.cholqr(ctx, d, passes=1, prec=eo.F32, M=m)
    assert int(info) == 0
    got = d.cpu().numpy()
    want = fp64_update(x, np.triu(z), True)
    fin = np.isfinite(want)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.array_equal(got[~fin & ~np.isnan(want)], want[~fin & ~np.isnan(want)].astype(np.float32))
    scale = np.where(np.isfinite(x), np.abs(x), 0).max(1)[:, None] * np.abs(z).max(0)[None, :]
    assert np.all(np.abs(got[fin] - want[fin]) <= 2.0 ** -23 * np.abs(want[fin]) + k * 2.0 ** -48 * scale[fin])


@pytest.mark.parametrize("k", [9, 16, 31])
def test_values_far_below_their_row(eo, ctx, k):
    """M = I given: X is returned as it is, to the smallest subnormal."""
    g = synth.rng(6700 + k)
    n = 20_003
    x = np.ldexp(g.uniform(0.5, 1.0, (n, k)), g.integers(-148, 120, (n, k))).astype(np.float32)
    x[::3] = synth.gaussian(len(x[::3]), k, 6800)
    x[g.integers(0, n, 50), g.integers(0, k, 50)] = 0.0
    d = dev(x)
    _, _, info = eo.cholqr(ctx, d, passes=1, prec=eo.F32, M=(dev(np.eye(k)), dev(np.zeros((k, k)))))
    assert int(info) == 0
    assert np.array_equal(d.cpu().numpy(), x)


@pytest.mark.parametrize("method", ["cholqr", "svqb"])
@pytest.mark.parametrize("decades", [-30, -24, -16, -8, 8, 16, 24, 30])
@pytest.mark.parametrize("k", [9, 16, 32])
def test_columns_of_widely_different_norms(eo, ctx, method, decades, k):
    """Columns of norms spread over the FP32 range, falling and rising, otherwise
    well conditioned.  Q is R^-1 of FP64 applied to X and rounded to FP32: every
    entry to 2^-23 and 2^-30 of its column's largest (R^-1 is formed here in FP64).
    SVQB's rank counts the eigenvalues above k 2^-52 of the largest."""
    n = 20_000
    s = 10.0 ** (np.linspace(0, decades, k) - min(decades, 0) * 0.5 - max(decades, 0) * 0.5)
    x = (synth.conditioned(n, k, 3.0, 6900 + k) * s).astype(np.float32)
    d = dev(x)
    if method == "cholqr":
        rh, _, info = eo.cholqr(ctx, d, passes=1, prec=eo.F32)
        assert int(info) == 0
        q = d.double().cpu().numpy()
        want = fp64_update(x, np.linalg.inv(rh.cpu().numpy()), True)
        assert np.max(np.abs(q.T @ q - np.eye(k))) <= 2.0 ** -18
        assert np.all(np.abs(q - want) <= 2.0 ** -23 * np.abs(want) + 2.0 ** -30 * np.abs(want).max(0))
    else:
        _, _, rank = eo.svqb(ctx, d, passes=1, prec=eo.F32)
        lam = np.linalg.svd(x.astype(np.float64), compute_uv=False) ** 2
        assert int(rank) <= np.sum(lam > 0.5 * k * 2.0 ** -52 * lam[0]) and int(rank) >= np.sum(lam > 2 * k * 2.0 ** -52 * lam[0])
        assert np.all(np.isfinite(d.cpu().numpy()))
