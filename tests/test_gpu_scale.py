"""Solves with sources of very small norm (needs a GB300): the Gram products' pivots have squared moduli near or
just above the smallest normal number (whose reciprocals are infinite).  The method is linear in B, so a power of two in B is one in X, up to what the
subnormal squares lose (they keep 40 bits here): the solutions agree to the tolerance of the solve."""
import pytest

from oracle import operator as O
from oracle import solver as S
from paper_0907_3261_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [1, 4])
@pytest.mark.parametrize("exponent", [0, -250, -255, -258, -261])
def test_solve_with_small_sources(L, exponent):
    import paper_0907_3261_gb300 as wd
    dims = (4, 4, 4, 4)
    links = I.random_links(dims, 0.3, seed=0)
    op = O.WilsonClover(links, dims, 0.115, 1.0)
    B = I.z4_noise(dims, L, seed=1)
    ctx = wd.wd_create(torch.from_numpy(links).cuda(), dims, 0.115, 1.0)
    X, info = wd.bbicggr_solve(ctx, torch.from_numpy(B * 2.0 ** exponent).cuda(), j=4, tol=1e-6, max_restarts=0)
    assert info["status"] == wd.WD_OK
    assert S.true_residual(op, B, X.cpu().numpy() * 2.0 ** -exponent).max() <= 1e-6
    wd.wd_destroy(ctx)
