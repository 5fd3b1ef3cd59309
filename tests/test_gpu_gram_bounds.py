"""What the tensor-core Gram engine promises at the ends of its range: totals
of many rows in one CTA, the error of short products, and columns whose first
rows are subnormal."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(np.asarray(a).T)).cuda().t()


@pytest.mark.parametrize("k", [1, 2, 4, 8])
def test_many_rows_in_one_cta(eo, tmp_path, k):
    """Products of up to 8 columns hold 16, 8, 4 or 2 parts of the rows side by
    side.  One CTA over 2^26 / 2^25 / 2^24 / 2^23 rows, 2^22 a part, its first
    panels at 1/4 and everything after them just below 2 (the two binades of
    headroom of the alignment exponent used up): the parts' sums together pass
    2^127 units.  The squared norms are summed exactly here, and q = x / |x| is
    rounded once (2 ulps)."""
    import torch

    np_ = 16 >> {1: 0, 2: 1, 4: 2, 8: 3}[k]
    q = 1 << 22
    n = np_ * q
    v = 2.0 - 2.0 ** -52
    x = torch.full((k, np_, q), v, dtype=torch.float64, device="cuda")
    x[:, :, :512] = 0.25
    if k > 1:  # signs of a Hadamard pattern (period 8) make the columns orthogonal
        s = torch.ones((k, 8), dtype=torch.float64)
        for c in range(k):
            for r in range(8):
                s[c, r] = -1.0 if bin(c & r).count("1") % 2 else 1.0
        x = (x.view(k, -1, 8) * s.cuda()[:, None, :]).view(k, np_, q)
    x = x.view(k, n)
    want = [0.25, v]
    norm2 = np_ * (512 * 0.25 ** 2 + (q - 512) * v * v)
    props = torch.cuda.get_device_properties(0)
    path = tmp_path / "tiles.txt"
    path.write_text("%d %d %d 1 0 %s/%d\n" % (k, n.bit_length() - 1, eo.DD, props.name.replace(" ", "_"),
                                             props.multi_processor_count))
    c = eo.Context(0)
    c.tune_cache(str(path))
    b = eo.Batch(c, [x.t()], passes=1, prec=eo.DD)
    assert b.tile(0)[0] == 1
    b.run()
    torch.cuda.synchronize()
    assert int(b.out[0]) == k
    for at, w in ((0, want[0]), (511, want[0]), (512, want[1]), (n - 1, want[1])):
        got = x[:, at].abs().cpu().numpy()
        assert np.all(np.abs(got * np.sqrt(norm2) / w - 1) <= 2.0 ** -50), (at, got)
    b.close()
    c.close()


@pytest.mark.parametrize("n", [1, 2, 4, 16, 63, 64, 65, 300])
@pytest.mark.parametrize("k", [1, 3, 4, 8, 12, 16, 17, 40])
def test_short_products(eo, ctx, monkeypatch, n, k):
    """Values over 20 binades below a column maximum of 1.  A product is off by
    less than 2^-105.7 (the dropped digit pairs and truncated values, see
    umma_gram.cu) and the result is rounded to a double-double (2^-106)."""
    monkeypatch.setenv("EO_DD_GRAM_ENGINE", "umma")
    g = synth.rng(3100 + 17 * n + k)

    def block(c):
        x = g.uniform(0.5, 1.0, (n, c)) * np.ldexp(1.0, -g.integers(0, 21, (n, c)))
        return np.asfortranarray(x / x.max(0) * np.where(g.random((n, c)) < 0.5, -1.0, 1.0))

    x = block(k)
    for y in (None, block(max(1, k // 2))):
        gh, gl = eo.gram(ctx, dev(x), None if y is None else dev(y))
        rh, rl = oracle.gram(x, y)
        err = np.abs((gh.cpu().numpy() - rh) + (gl.cpu().numpy() - rl))
        assert np.all(err <= 2.0 ** -105 * np.abs(rh) + n * 2.0 ** -105), float(np.log2(err.max() / n))


@pytest.mark.parametrize("n,kx,ky", [(300_000, 16, 0), (300_000, 9, 5), (200_000, 40, 17), (1_200_000, 4, 0), (600_000, 8, 0)])
def test_columns_that_begin_with_subnormals(eo, ctx, n, kx, ky):
    """A column whose first panels hold subnormals only: they stand on the grid of
    exponent 1 and are shifted like any others when the first normal value
    raises the column's exponent."""
    x = synth.gaussian(n, kx, 3300 + kx)
    y = synth.gaussian(n, ky, 3400 + ky) if ky else None
    for a in (x, y) if ky else (x,):
        a[:600, -1] *= 2e-309
        a[:600, 0] = 0.0
        a[100:110, 0] = 5e-324
    gh, gl = eo.gram(ctx, dev(x), None if y is None else dev(y))
    rh, rl = oracle.gram(x, y)
    y = x if y is None else y
    err = np.abs((gh.cpu().numpy() - rh) + (gl.cpu().numpy() - rl))
    tol = 2.0 ** -104 * np.abs(rh) + n * 2.0 ** -103 * np.outer(np.abs(x).max(0), np.abs(y).max(0))
    assert np.all(err <= tol), float((err / tol).max())


@pytest.mark.parametrize("n,kx,ky", [(2_000_000, 64, 16), (4_000_000, 16, 0), (8_000_000, 4, 0)])
def test_zeros_cost_little(eo, ctx, n, kx, ky):
    """A zero column, and every thousandth value zero: within half of the dense
    product's time (measured: 4 %)."""
    import torch

    g = torch.Generator(device="cuda")
    g.manual_seed(3500 + kx)
    x = torch.randn((kx, n), generator=g, device="cuda", dtype=torch.float64)
    y = torch.randn((ky, n), generator=g, device="cuda", dtype=torch.float64).t() if ky else None

    def best(a):
        times = []
        for _ in range(8):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            eo.gram(ctx, a.t(), y)
            t1.record()
            torch.cuda.synchronize()
            times.append(t0.elapsed_time(t1))
        return min(times[2:])

    dense = best(x)
    x[:, torch.rand(n, generator=g, device="cuda") < 1e-3] = 0.0
    rare = best(x)
    x[kx - 1] = 0.0
    assert max(rare, best(x)) <= 1.5 * dense


@pytest.mark.parametrize("rate", [2e-5, 1e-3])
@pytest.mark.parametrize("kx,ky", [(64, 16), (40, 9), (20, 4), (16, 16), (16, 0), (4, 0)])
@pytest.mark.parametrize("odd_ld", [False, True])
def test_panels_of_every_kind_in_turn(eo, ctx, kx, ky, rate, odd_ld):
    """Many panels a CTA: near ones, ones with values below the near window (all
    digits, in steps), with zeros, and with growing exponents, in random order."""
    import torch

    n = 500_003
    g = synth.rng(3600 + kx)

    def block(k, seed):
        a = synth.gaussian(n, k, seed)
        m = g.random(a.shape) < rate
        a[m] *= np.ldexp(1.0, -g.integers(20, 110, int(m.sum())))
        a[g.random(a.shape) < rate] = 0.0
        for i in range(40):
            a[g.integers(0, n), g.integers(0, k)] *= 2.0 ** g.integers(2, 9)
        return a

    def put(a):
        ld = n + 1 if not odd_ld else n
        t = torch.full((a.shape[1], ld), float("nan"), dtype=torch.float64, device="cuda")
        t[:, :n] = torch.from_numpy(np.ascontiguousarray(a.T))
        return t.t()[:n]

    x = block(kx, 3700 + kx)
    y = block(ky, 3800 + ky) if ky else None
    gh, gl = eo.gram(ctx, put(x), None if y is None else put(y))
    rh, rl = oracle.gram(x, y)
    y = x if y is None else y
    err = np.abs((gh.cpu().numpy() - rh) + (gl.cpu().numpy() - rl))
    tol = 2.0 ** -104 * np.abs(rh) + n * 2.0 ** -103 * np.outer(np.abs(x).max(0), np.abs(y).max(0))
    assert np.all(err <= tol), float((err / tol).max())
