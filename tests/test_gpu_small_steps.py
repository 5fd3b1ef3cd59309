"""The k-by-k steps of the compensated modes (Cholesky and Jacobi in 128-bit
floating point) at the edges of their sizes -- one column, odd and even counts,
a full 64 -- against the binary128 oracle, on the same Gram matrix.

Given M, both sides factor it with relative errors far below 2^-104, so R and Z
differ by at most about kappa(M) k 2^-104 of their size (kappa(M) =
kappa(X)^2) plus the rounding of the double-double results."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

U, U2 = 2.0 ** -53, 2.0 ** -104


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(np.asarray(a).T)).cuda().t()


def close(hi, lo, ref_hi, ref_lo, tol):
    err = np.abs((hi.cpu().numpy() - ref_hi) + (lo.cpu().numpy() - ref_lo))
    assert np.max(err) <= tol * np.max(np.abs(ref_hi)), float(np.max(err) / (tol * np.max(np.abs(ref_hi))))


@pytest.mark.parametrize("prec", [1, 3])
@pytest.mark.parametrize("k,kappa", [(1, 1.0), (2, 1e9), (3, 1e3), (15, 1e6), (16, 1e10), (31, 1e5), (33, 1e8), (64, 1e4)])
def test_cholesky_and_jacobi_of_a_given_gram_matrix(eo, ctx, prec, k, kappa):
    n = 700
    x = synth.conditioned(n, k, kappa, 5100 + k)
    mh, ml = oracle.gram(x)
    tol = 64 * k * kappa ** 2 * U2
    d = dev(x)
    rh, rl, info = eo.cholqr(ctx, d, prec=prec, M=(dev(mh), dev(ml)))
    q_o, (rh_o, rl_o), info_o = oracle.cholqr(x, m=(mh, ml))
    assert int(info.item()) == info_o == 0
    close(rh, rl, rh_o, rl_o, tol)
    assert np.max(np.abs(d.cpu().numpy() - q_o)) <= tol + 4 * U
    d = dev(x)
    zh, zl, rank = eo.svqb(ctx, d, prec=prec, M=(dev(mh), dev(ml)))
    q_o, (zh_o, zl_o), rank_o = oracle.svqb(x, m=(mh, ml))
    assert int(rank.item()) == rank_o == k
    close(zh, zl, zh_o, zl_o, tol)
    assert np.max(np.abs(d.cpu().numpy() - q_o)) <= tol + 4 * U
    z = zh.cpu().numpy()
    assert np.array_equal(z, z.T)


@pytest.mark.parametrize("k", [2, 7, 16, 33])
def test_exactly_dependent_columns(eo, ctx, k):
    """A repeated column: CholQR reports it and leaves X, SVQB counts the rank."""
    x = np.round(synth.gaussian(500, k, 5200 + k) * 64)
    x[:, k - 1] = 3 * x[:, 0]
    d = dev(x)
    _, _, info = eo.cholqr(ctx, d, prec=eo.DD)
    assert int(info.item()) == k
    assert np.array_equal(d.cpu().numpy(), x)
    _, _, rank = eo.svqb(ctx, dev(x), prec=eo.DD)
    assert int(rank.item()) == k - 1


def test_graded_columns_keep_their_relative_accuracy(eo, ctx):
    """Columns of norms 1 .. 1e-12, otherwise well conditioned: the eigenvalues
    of M span 24 decades and Z is still accurate to its smallest entries' size."""
    n, k = 900, 12
    s = 10.0 ** -np.arange(k)
    x = synth.conditioned(n, k, 3.0, 5300) * s
    d = dev(x)
    zh, zl, rank = eo.svqb(ctx, d, prec=eo.DD, tol=0.0)
    q_o, (zh_o, zl_o), rank_o = oracle.svqb(x, tol=0.0)
    assert int(rank.item()) == rank_o == k
    assert oracle.orth_err(np.asfortranarray(d.cpu().numpy()))[0] <= 1e-14
    assert np.max(np.abs(d.cpu().numpy() - q_o)) <= 1e-13
