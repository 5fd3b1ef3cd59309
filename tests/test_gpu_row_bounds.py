"""The tensor-core row engine at its own bound: Y is the product V C rounded to
FP64, so Y - V C leaves 2^-53 of it and its FP64 rounding shows errors of 2^-106.

A product is off by less than 2^-103 of the row's and the column's largest
values (dropped digit pairs) and by 2^-108 and 2^-109 (truncation of C and V,
umma_rowprod.cu): 2^-102 of them, kv times, is tested, and one rounding."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(np.asarray(a).T)).cuda().t()


@pytest.mark.parametrize("kv,k", [(9, 5), (16, 16), (20, 4), (32, 32), (40, 12), (64, 16)])
@pytest.mark.parametrize("spread", [0, 20, 40, 90])
def test_residual_of_a_rounded_product(eo, ctx, monkeypatch, kv, k, spread):
    monkeypatch.setenv("EO_DD_ROW_ENGINE", "umma")
    n = 3_001
    g = synth.rng(7100 + kv + spread)
    v = g.uniform(0.5, 1.0, (n, kv)) * np.where(g.random((n, kv)) < 0.5, -1.0, 1.0)
    ch = np.asfortranarray(g.standard_normal((kv, k)))
    if spread:
        v *= np.ldexp(1.0, -g.integers(0, spread + 1, (n, kv)))
        ch *= np.ldexp(1.0, -g.integers(0, spread + 1, (kv, k)))
    v = np.asfortranarray(v)
    cl = np.asfortranarray(ch * 2.0 ** -55 * g.uniform(-1, 1, (kv, k)))
    y = -oracle.project_apply(v, np.zeros((n, k), order="F"), ch, cl)
    out, _ = eo.project_apply(ctx, dev(v), dev(y), (dev(ch), dev(cl)), prec=eo.DD, want_m=False)
    ref = oracle.project_apply(v, y, ch, cl)
    scale = np.abs(v).max(1)[:, None] * (np.abs(ch) + np.abs(cl)).max(0)[None, :]
    err = np.abs(out.cpu().numpy() - ref)
    tol = 2 * U * np.abs(ref) + kv * 2.0 ** -102 * scale
    assert np.all(err <= tol), float(np.log2((err / scale).max() / kv))
