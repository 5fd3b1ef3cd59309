"""CholQR and SVQB with a Gram matrix given by the caller."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(np.asarray(a).T)).cuda().t()


@pytest.mark.parametrize("prec", ["FP64", "F32"])
@pytest.mark.parametrize("low", [np.nan, np.inf, 1e300])
def test_low_parts_are_not_read_in_fp64(eo, ctx, prec, low):
    """FP64 factorizations take the high part of M alone: what stands in the low
    part changes nothing, bit for bit."""
    p = getattr(eo, prec)
    x = synth.gaussian(3_000, 6, 6100)
    x = x.astype(np.float32) if prec == "F32" else x
    mh, _ = eo.gram(ctx, dev(x), prec=p)
    for f in (eo.cholqr, eo.svqb):
        out = []
        for lo in (np.zeros((6, 6)), np.full((6, 6), low)):
            d = dev(x)
            h, _, flag = f(ctx, d, prec=p, M=(mh, dev(lo)))
            out.append((int(flag), h.cpu().numpy(), d.cpu().numpy()))
        assert out[0][0] == out[1][0] == (0 if f is eo.cholqr else 6)
        assert np.array_equal(out[0][1], out[1][1]) and np.array_equal(out[0][2], out[1][2])
