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


def indefinite(kind, k):
    g = synth.rng(6200 + k)
    if kind == "zero pivot":  # a leading block of ones leaves a zero diagonal with entries beside it
        m = np.ones((k, k))
        m[1, 2] = m[2, 1] = 2.0
        m[np.arange(3, k), np.arange(3, k)] = 5.0 + np.arange(k - 3)
        return m
    a = g.integers(-8, 9, (k, k)).astype(float)
    m = a + a.T
    if kind == "hollow":
        m[np.arange(k), np.arange(k)] = 0.0
    else:  # two rows with a zero diagonal beside a definite block
        m = a @ a.T + np.diag(np.arange(k) + 1.0)
        m[k - 2:, :] = m[:, k - 2:] = 0.0
        m[k - 2, k - 1] = m[k - 1, k - 2] = 3.0
    return m


@pytest.mark.parametrize("prec", [1, 3])
@pytest.mark.parametrize("kind,k", [("zero pivot", 3), ("zero pivot", 8), ("hollow", 2), ("hollow", 7), ("hollow", 33),
                                    ("block", 4), ("block", 17)])
def test_svqb_of_an_indefinite_matrix(eo, ctx, prec, kind, k):
    """A given M that is not semidefinite, with diagonal entries that are zero or
    become zero in the elimination: Z keeps the positive eigenvalues, as the
    oracle's does.  (Eigenvalues of matrices of small integers, apart by more than
    2^-20 of their size: 2^-70 is a wide tolerance.)"""
    m = indefinite(kind, k)
    lam = np.linalg.eigvalsh(m)
    assert lam[0] < -0.1 and np.min(np.abs(lam)) > 1e-6 * lam[-1]
    x = synth.gaussian(300, k, 6300 + k)
    d = dev(x)
    zh, zl, rank = eo.svqb(ctx, d, prec=prec, M=(dev(m), dev(0 * m)))
    q_o, (zh_o, zl_o), rank_o = oracle.svqb(x, m=(m, 0 * m))
    assert int(rank) == rank_o == int(np.sum(lam > 0))
    err = (zh.cpu().numpy() - zh_o) + (zl.cpu().numpy() - zl_o)
    assert np.max(np.abs(err)) <= 2.0 ** -70 * np.max(np.abs(zh_o))
    assert np.max(np.abs(d.cpu().numpy() - q_o)) <= 1e-13 * np.max(np.abs(q_o))
