"""The block updates in exact digits, element by element (needs a GB300): blocks whose columns or entries span
twenty orders of magnitude, with matrices that do not make up for it, keep every element's own accuracy.

Bounds: a sum of L products in FP64 is off by at most 2 (L + 2) U of the sum of the terms' moduli, U = 2^-53;
in double-float arithmetic (precision 1) U is 2^-44, what FP32 pairs keep of a term after a sum's renormalisations.
The digits are off by 2^-50 of the largest factors' product in seven and 2^-58 in eight, and an element whose
largest term is below 2^-9 of that product is computed in FP64."""
import numpy as np
import pytest

from paper_0907_3261_gb300 import inputs as I
from test_gpu_digits import context, dev, host, wide

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wd():
    import paper_0907_3261_gb300 as wd
    return wd


def unit(L, precision):
    return 2 * (L + 2) * (2.0 ** -53 if precision == 0 else 2.0 ** -44)


def matrix(kind, L, rng):
    c = rng.normal(size=(L, L)) + 1j * rng.normal(size=(L, L))
    if kind == "identity":
        return np.eye(L, dtype=complex)
    if kind == "diagonal":
        return np.diag(np.diag(c)).copy()
    if kind == "upper":
        return np.triu(c)
    if kind == "lower":
        return np.tril(c)
    if kind == "nearly diagonal":
        return np.diag(np.diag(c)) + 2.0 ** -10 * c
    if kind == "tiny":
        return c * 10.0 ** rng.integers(-310, -290, size=(L, L))
    return c


def blocks(kind, n, L, rng, count):
    out = []
    for _ in range(count):
        b = rng.normal(size=(n, L)) + 1j * rng.normal(size=(n, L))
        if kind == "columns":
            b *= 10.0 ** -np.linspace(0, 20, L)
        elif kind == "entries":
            b *= 2.0 ** rng.integers(-60, 1, size=(n, L))
        elif kind == "points":
            b *= rng.random((n, L)) < 0.05
        out.append(b)
    return out


MATRICES = ["identity", "diagonal", "upper", "lower", "nearly diagonal", "dense", "tiny"]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("spread", ["none", "columns", "entries", "points"])
@pytest.mark.parametrize("dims,L", [((3, 3, 3, 3), 2), ((2, 3, 2, 5), 4), ((3, 3, 3, 5), 7), ((4, 4, 4, 4), 12),
                                    ((3, 3, 5, 3), 16)])
def test_products(wd, dims, L, spread, precision):
    rng = np.random.default_rng(L)
    n = 12 * int(np.prod(dims))
    ctx = context(wd, dims)
    eps = unit(L, precision)
    z = 0.3 - 0.7j
    for kind in MATRICES:
        P, V, R, W, U, Y, Rt = (b.reshape(-1, 12, L) for b in blocks(spread, n, L, rng, 7))
        c = matrix(kind, L, rng)
        cw, ca = c.astype(np.clongdouble), np.abs(c)
        low = 2.0 ** -1070                                # where FP64 itself underflows
        u = dev(np.zeros_like(P))
        wd.bb_update_u(ctx, dev(P), dev(V), u, z, c, precision=precision)
        mod = np.abs(wide(P, L)) + abs(z) * np.abs(wide(V, L))
        err = np.abs(wide(host(u), L) - (wide(P, L) - np.clongdouble(z) * wide(V, L)) @ cw)
        assert (err <= eps * (mod @ ca) + low).all(), kind
        p, v = dev(np.zeros_like(P)), dev(np.zeros_like(P))
        wd.bb_update_pv(ctx, p, v, dev(R), dev(W), dev(U), dev(Y), dev(Rt), c, precision=precision)
        for got, base, A in ((p, R, U), (v, W, Y)):
            ref = wide(base, L) + wide(A, L) @ cw
            lim = eps * (np.abs(wide(A, L)) @ ca) + 2.0 ** -52 * np.abs(wide(base, L)) + low
            assert (np.abs(wide(host(got), L) - ref) <= lim).all(), kind
    wd.wd_destroy(ctx)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("spread", ["none", "columns", "entries", "points", "where the other is small"])
@pytest.mark.parametrize("dims,L", [((3, 3, 3, 3), 2), ((2, 3, 2, 5), 4), ((3, 3, 3, 5), 7), ((4, 4, 4, 4), 12),
                                    ((3, 3, 5, 3), 16)])
def test_gram_products(wd, dims, L, spread, precision):
    """R~^H V with V = W (gamma = 0) and R~^H R with R unchanged (zeta = 0, Y = 0).  A tile of 16 rows adds at most
    2 U a row of the terms' moduli, and its sums are added up a few at a time: 64 U in all."""
    rng = np.random.default_rng(L)
    n = 12 * int(np.prod(dims))
    A, B = blocks("none" if spread[0] == "w" else spread, n, L, rng, 2)
    if spread[0] == "w":
        few = rng.random((n, 1)) < 0.02                  # rows of R~ that are not zero, where the other block is small
        A, B = A * few, B * np.where(few, 1e-13, 1.0)
        A[::37] *= 1e-290
        A[5] = 1e-315
    ctx = context(wd, dims)
    lim = 64 * (2.0 ** -53 if precision == 0 else 2.0 ** -44) * (np.abs(A).T @ np.abs(B)) + 2.0 ** -1060
    ref = A.astype(np.clongdouble).conj().T @ B.astype(np.clongdouble)
    a, b = (dev(x.reshape(-1, 12, L)) for x in (A, B))
    zero, out = dev(np.zeros((n // 12, 12, L), complex)), dev(np.zeros((n // 12, 12, L), complex))
    none = np.zeros((L, L), complex)
    got = wd.bb_update_pv(ctx, out, zero.clone(), b, b, b, b, a, none, precision=precision)
    assert (np.abs(got - ref) <= lim).all()
    got, norms = wd.bb_update_xr(ctx, out, zero, zero, b, zero, zero, a, 0.0, precision=precision)
    assert (np.abs(got - ref) <= lim).all()
    wd.wd_destroy(ctx)
