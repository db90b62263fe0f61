"""The block updates in exact digits (bb_update_u, bb_update_xr, bb_update_pv) against extended precision:
every group count of columns and its remainders, rows that do not fill a tile, columns of very different
size, and infinities and NaNs.

Bounds: a factor is held to 2^-54 (seven digits; 2^-62 with eight, which precision 0 takes below L = 4) of a
scale that is at most four times the largest factor of its row or column, so a term of a product is off by
at most 2^-50 (2^-58) of the largest factors' product; FP64 sums and roundings add a few 2^-53 of the terms'
moduli.
"""
import numpy as np
import pytest

from paper_0907_3261_gb300 import inputs as I

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def wd():
    import paper_0907_3261_gb300 as wd
    return wd


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    return t.cpu().numpy()


def wide(a, L):
    return a.reshape(-1, L).astype(np.clongdouble)


def product_bound(A, C, eps):
    """Per element of A C: the terms' moduli times 16 U, and 2 L eps of the largest factors after the rows of C
    have been scaled to one."""
    L = C.shape[0]
    r = np.abs(C).max(axis=1)
    r[r == 0] = 1
    big = (np.abs(A) * r).max(axis=1)[:, None] * (np.abs(C) / r[:, None]).max(axis=0)[None, :]
    return 16 * U * (np.abs(A) @ np.abs(C)) + 2 * L * eps * big


def case(dims, L, seed, spread):
    n = 12 * int(np.prod(dims))
    rng = np.random.default_rng(seed)
    blocks = [(rng.normal(size=(n, L)) + 1j * rng.normal(size=(n, L))) for _ in range(9)]
    c = rng.normal(size=(L, L)) + 1j * rng.normal(size=(L, L))
    if spread:
        # columns of the direction blocks from 1e-12 to 1, the matrix's rows the other way round
        s = 10.0 ** -np.linspace(0, 12, L)
        blocks = [b * s for b in blocks]
        c = c / s[:, None] * s[None, :]
    return [b.reshape(-1, 12, L) for b in blocks], c


def context(wd, dims):
    return wd.wd_create(dev(I.random_links(dims, 0.2, seed=0)), dims, 0.12, 1.0)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("spread", [False, True])
@pytest.mark.parametrize("dims,L", [((2, 2, 2, 3), 1), ((2, 2, 2, 2), 3), ((3, 2, 3, 3), 4), ((3, 3, 3, 3), 5),
                                    ((2, 3, 2, 5), 8), ((3, 3, 3, 5), 9), ((4, 4, 4, 4), 12),
                                    ((3, 3, 5, 3), 13), ((4, 4, 4, 6), 16)])
def test_updates_in_digits(wd, dims, L, spread, precision):
    (P, V, X, F, G, R, W, Y, Rt), c = case(dims, L, 100 * L + spread, spread)
    ctx = context(wd, dims)
    eps = 2.0 ** -58 if precision == 0 and L < 4 else 2.0 ** -50
    z = 0.3 - 0.7j
    cw = c.astype(np.clongdouble)

    u = dev(np.zeros_like(P))
    wd.bb_update_u(ctx, dev(P), dev(V), u, z, c, precision=precision)
    S = wide(P, L) - np.clongdouble(z) * wide(V, L)
    lim = product_bound(np.abs(P.reshape(-1, L)) + abs(z) * np.abs(V.reshape(-1, L)), c, eps)
    assert (np.abs(wide(host(u), L) - S @ cw) <= lim).all()

    def gram(got, A, B):
        A, B = wide(A, L), wide(B, L)
        lim = 2 * U * len(A) * np.abs(A).max(axis=0)[:, None] * np.abs(B).max(axis=0)[None, :]
        assert (np.abs(got - A.conj().T @ B) <= lim).all()

    x, r = dev(X), dev(R)
    rtr, nrm = wd.bb_update_xr(ctx, x, dev(F), dev(G), r, dev(W), dev(Y), dev(Rt), z, precision=precision)
    for got, t, f, g in ((x, X, F, G), (r, R, -W, -Y)):
        ref = wide(t, L) + np.clongdouble(z) * wide(f, L) + wide(g, L)
        lim = 6 * U * (np.abs(wide(t, L)) + 2 * abs(z) * np.abs(wide(f, L)) + np.abs(wide(g, L)))
        assert (np.abs(wide(host(got), L) - ref) <= lim).all()
    gram(rtr, Rt, host(r))
    n2 = (np.abs(wide(host(r), L)) ** 2).sum(axis=0)
    assert (np.abs(nrm - n2) <= U * r.numel() * n2).all()

    p, v = dev(np.zeros_like(P)), dev(np.zeros_like(P))
    rtv = wd.bb_update_pv(ctx, p, v, dev(R), dev(W), dev(P), dev(Y), dev(Rt), c, precision=precision)
    for got, base, A in ((p, R, P), (v, W, Y)):
        lim = product_bound(np.abs(A.reshape(-1, L)), c, eps) + 2 * U * np.abs(base.reshape(-1, L))
        assert (np.abs(wide(host(got), L) - wide(base, L) - wide(A, L) @ cw) <= lim).all()
    gram(rtv, Rt, host(v))
    wd.wd_destroy(ctx)


@pytest.mark.parametrize("precision", [0, 1])
def test_values_that_are_not_finite_and_zeros(wd, precision):
    dims, L = (2, 2, 3, 3), 6
    (P, V, X, F, G, R, W, Y, Rt), c = case(dims, L, 5, False)
    ctx = context(wd, dims)
    P.reshape(-1, L)[7, 2] = np.inf
    P.reshape(-1, L)[100, 5] = complex(0, np.nan)
    P.reshape(-1, L)[31] = 0
    V.reshape(-1, L)[31] = 0
    c[:, 4] = 0
    u = dev(np.ones_like(P))
    wd.bb_update_u(ctx, dev(P), dev(V), u, 0.5, c, precision=precision)
    got = host(u).reshape(-1, L)
    bad = np.zeros(len(got), bool)
    bad[[7, 100]] = True
    assert not np.isfinite(got[bad]).any() and np.isfinite(got[~bad]).all()
    assert (got[31] == 0).all() and (got[~bad, 4] == 0).all()

    # V = W + Y gamma with a NaN in one row of W: that column of R~^H V, and no other
    W.reshape(-1, L)[50, 1] = np.nan
    Rt.reshape(-1, L)[:, 3] = 0
    p, v = dev(np.zeros_like(P)), dev(np.zeros_like(P))
    rtv = wd.bb_update_pv(ctx, p, v, dev(R), dev(W), dev(Y), dev(Y), dev(Rt), c, precision=precision)
    assert not np.isfinite(rtv[:, 1]).any() and np.isfinite(np.delete(rtv, 1, axis=1)).all()
    assert (np.delete(rtv[3], 1) == 0).all()
    wd.wd_destroy(ctx)
