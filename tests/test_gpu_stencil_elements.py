"""The FP64 stencils element by element (needs a GB300): sites whose own components span many orders of magnitude
and lie far above their neighbours', sites far below them, and hopping parameters that make the neighbours'
part small.

Bounds per element, U = 2^-53: the site block's sum of 6 complex products in FP64, on both sides, 32 U of its terms'
moduli; the hopping sum, whose parts FP64 arithmetic rounds relative to themselves, 64 U |kappa| of the
neighbours' largest components (2 spins x 3 colours of unit links).  The two sides' site blocks agree to 16 U of
c_SW |kappa| (sums of 4 leaves), in every entry of a chirality."""
import numpy as np
import pytest

from oracle import operator as O
from oracle import solver as S
from paper_0907_3261_gb300 import inputs as I
from test_gpu_fixed import dev, host

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def wd():
    import __graft_entry__
    __graft_entry__.build()
    import paper_0907_3261_gb300 as pkg
    return pkg


def around(dims, x):
    """Largest modulus among the eight neighbours' components, [V][L]."""
    m = np.abs(x).reshape(dims[3], dims[2], dims[1], dims[0], 12, -1).max(axis=4)
    return np.max([np.roll(m, d, axis=a) for a in range(4) for d in (1, -1)], axis=0).reshape(-1, x.shape[-1])


def blocks_abs(blocks, extra, x):
    """sum_j (|B_ij| + extra) |x_j|, [V][12][L], `extra` within a chirality."""
    return (np.abs(blocks) + extra * np.kron(np.eye(2), np.ones((6, 6)))) @ np.abs(x)


def field(kind, dims, L, seed):
    rng = np.random.default_rng(seed)
    V = int(np.prod(dims))
    X = I.gaussian_block(dims, L, seed=seed).reshape(V, 12, L)
    high = rng.random((V, 1, L)) < 0.08
    if kind == "high sites":        # components from 1 to 1e-18 above a background of 1e-20
        own = 10.0 ** -rng.integers(0, 19, size=(V, 12, L))
        X = X * np.where(high, own, 1e-20)
    elif kind == "points":
        X = X * high * (rng.random((V, 12, L)) < 0.5)
    elif kind == "low sites":
        X = X * np.where(high, 1e-20, 1.0)
    return X


@pytest.mark.parametrize("kappa,csw", [(0.12, 0.0), (0.12, 1.0), (-0.2, 0.0), (0.0, 0.0), (1e-6, 0.0), (0.005, 0.0),
                                       (0.01, 0.0), (0.02, 0.0)])
@pytest.mark.parametrize("kind", ["gaussian", "high sites", "points", "low sites"])
@pytest.mark.parametrize("dims,L", [((4, 3, 5, 4), 2), ((4, 4, 4, 4), 5)])
def test_products_and_sweeps(wd, dims, L, kind, kappa, csw):
    links = I.random_links(dims, 0.3, seed=1)
    op = O.WilsonClover(links, dims, kappa, csw)
    ctx = wd.wd_create(dev(links), dims, kappa, csw)
    V = int(np.prod(dims))
    X = field(kind, dims, L, 3)
    shape = (V, 4, 3, L)

    def limit(blocks, v, hops):
        extra = 2 * csw * abs(kappa)
        return 32 * U * blocks_abs(blocks, extra, v) + 64 * U * abs(kappa) * hops[:, None]

    Y = host(wd.wd_apply(ctx, dev(X.reshape(shape)))).reshape(V, 12, L)
    ref = op.apply(X.reshape(shape)).reshape(V, 12, L)
    assert (np.abs(Y - ref) <= limit(op.AD, X, around(dims, X))).all()
    # G = A_D^{-1} (X + kappa H G), the last sweep's own roundings and those of G before it
    G1 = S.jacobi(op, X.reshape(shape), 1).reshape(V, 12, L)
    G = host(wd.jacobi_precond(ctx, dev(X.reshape(shape)), 2)).reshape(V, 12, L)
    ref = S.jacobi(op, X.reshape(shape), 2).reshape(V, 12, L)
    hops = around(dims, G1)
    inner = np.abs(X) + 16 * abs(kappa) * hops[:, None]
    lim = limit(op.AD_inv, inner, hops) + blocks_abs(op.AD_inv, 0, np.broadcast_to(64 * U * abs(kappa) * hops[:, None], X.shape))
    assert (np.abs(G - ref) <= lim).all()
    wd.wd_destroy(ctx)
