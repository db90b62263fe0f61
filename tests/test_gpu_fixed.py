"""The fixed-point form of the FP64 stencils (csrc/dslash_fx.cu) at the edges of its dispatch (needs a
GB300): columns read through L1 (L = 1, 2) and staged (L >= 3), CTAs that end inside a site or a
lattice, site blocks and kappa of extreme scales, capture before its workspace exists.

Tolerance: the fixed-point sums are exact to 2^-57 of their bound, but the site blocks and their
inverses come from FP64 arithmetic on both sides (a few 2^-53), as does the oracle's own product:
60 products of at most the bound each, 60 * 2^-53 ~ 7e-15, stays below 1e-14 of the bound
|A|_inf max|X| (tests/test_gpu_x3.py uses the same reasoning with the largest output as the bound)."""
import numpy as np
import pytest

from oracle import operator as O
from oracle import solver as S
from paper_0907_3261_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-14


@pytest.fixture(scope="module")
def wd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_0907_3261_gb300 as pkg
    return pkg


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy()


def block_bound(blocks):
    return np.abs(blocks).sum(axis=-1).max()


@pytest.mark.parametrize("dims,L", [((2, 2, 2, 2), 1), ((3, 5, 2, 7), 1), ((5, 3, 4, 3), 2),
                                    ((3, 5, 2, 7), 3), ((3, 3, 3, 5), 4), ((7, 2, 3, 3), 13),
                                    ((2, 3, 2, 2), 16), ((8, 8, 8, 8), 11)])
def test_products_and_sweeps_at_the_edges(wd, dims, L):
    links = I.random_links(dims, 0.3, seed=sum(dims) + L)
    X = I.gaussian_block(dims, L, seed=4)
    op = O.WilsonClover(links, dims, 0.125, 1.1)
    ctx = wd.wd_create(dev(links), dims, 0.125, 1.1)
    assert wd.wd_get_apply_form(ctx) == 1
    bound = (block_bound(op.AD) + 16 * 0.125) * np.abs(X).max()
    assert np.abs(host(wd.wd_apply(ctx, dev(X))) - op.apply(X)).max() <= TOL * bound
    for j in (2, 3):
        G, Go = host(wd.jacobi_precond(ctx, dev(X), j)), S.jacobi(op, X, j)
        inv = block_bound(op.AD_inv)
        assert np.abs(G - Go).max() <= j * TOL * inv * (1 + 16 * 0.125 * inv) ** (j - 1) * np.abs(X).max()


@pytest.mark.parametrize("kappa,csw", [(0.0, 1.0), (1e-6, 1.0), (-0.13, 1.0), (0.9, 0.3), (7.0, 0.02),
                                       (0.04, 60.0), (0.13, 900.0)])
def test_scales_of_kappa_and_of_the_site_blocks(wd, kappa, csw):
    dims, L = (4, 3, 2, 5), 5
    links = I.random_links(dims, 0.2, seed=2)
    X = I.gaussian_block(dims, L, seed=3)
    op = O.WilsonClover(links, dims, kappa, csw)
    ctx = wd.wd_create(dev(links), dims, kappa, csw)
    assert wd.wd_get_apply_form(ctx) == 1
    bound = (block_bound(op.AD) + 16 * abs(kappa)) * np.abs(X).max()
    assert np.abs(host(wd.wd_apply(ctx, dev(X))) - op.apply(X)).max() <= TOL * bound


@pytest.mark.parametrize("j", [-900, 900])
def test_sweeps_scale_exactly_up_to_the_ends_of_the_range(wd, j):
    dims = (4, 4, 2, 3)
    ctx = wd.wd_create(dev(I.random_links(dims, 0.3, seed=1)), dims, 0.12, 1.0)
    R = I.gaussian_block(dims, 4, seed=2)
    G = host(wd.jacobi_precond(ctx, dev(R), 4))
    Y = host(wd.wd_apply(ctx, dev(R)))
    assert np.array_equal(host(wd.jacobi_precond(ctx, dev(R * 2.0 ** j), 4)), G * 2.0 ** j)
    assert np.array_equal(host(wd.wd_apply(ctx, dev(R * 2.0 ** j))), Y * 2.0 ** j)


@pytest.mark.parametrize("L", [2, 6])
def test_sweeps_with_zero_and_non_finite_columns(wd, L):
    dims = (3, 4, 5, 2)
    V = int(np.prod(dims))
    ctx = wd.wd_create(dev(I.random_links(dims, 0.3, seed=1)), dims, 0.12, 1.0)
    R = I.gaussian_block(dims, L, seed=2)
    clean = host(wd.jacobi_precond(ctx, dev(R), 3))
    R[..., 0] = 0.0
    R.reshape(V, 12, L)[7, 5, 1] = np.inf
    G = host(wd.jacobi_precond(ctx, dev(R), 3)).reshape(V, 12, L)
    assert np.array_equal(G[..., 0], np.zeros((V, 12)))
    assert not np.isfinite(G[7, :, 1]).any() and not np.isfinite(G[..., 1]).all()
    assert np.array_equal(G[..., 2:], clean.reshape(V, 12, L)[..., 2:])


def test_first_product_under_capture_uses_the_fp64_pipe(wd):
    """A capture cannot allocate the operand's copy, so the product runs on the FP64 pipe, as with
    wd_set_apply_form 0; after a product outside the capture it runs in fixed point."""
    dims, L = (4, 4, 4, 4), 3
    links, X = I.random_links(dims, 0.3, seed=1), I.gaussian_block(dims, L, seed=2)
    ctx = wd.wd_create(dev(links), dims, 0.12, 1.0)
    x = dev(X)
    wd.wd_set_apply_form(ctx, 0)
    pipe = host(wd.wd_apply(ctx, x))
    wd.wd_set_apply_form(ctx, 1)

    def captured():
        y, g, s = torch.empty_like(x), torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(g, stream=s):
            wd.wd_apply(ctx, x, y, stream=s)
        g.replay()
        return host(y)

    assert np.array_equal(captured(), pipe)
    fixed = host(wd.wd_apply(ctx, x))
    assert np.array_equal(captured(), fixed)
