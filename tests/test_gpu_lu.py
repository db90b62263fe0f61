"""The L x L solves for alpha and gamma through whole solves against the oracle: one element per thread,
so block widths whose 2 L^2 elements fill their warps or do not, the smallest and the largest.

Bounds: the iterates solve the same recurrences in FP64, so the iteration counts agree to 2 and the
solutions, both with true residuals below 1e-12, to 1e-10.
"""
import numpy as np
import pytest

from oracle import operator as O
from oracle import solver as S
from paper_0907_3261_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [1, 2, 4, 5, 7, 11, 13, 16])
def test_solves_of_every_block_width_match_the_oracle(L):
    import torch
    import paper_0907_3261_gb300 as wd
    dims = (4, 4, 4, 4)
    links = I.random_links(dims, 0.3, seed=0)
    op = O.WilsonClover(links, dims, 0.115, 1.0)
    B = I.gaussian_block(dims, L, seed=L)
    ref = S.solve(op, B, j=2, tol=1e-12)
    ctx = wd.wd_create(torch.from_numpy(links).cuda(), dims, 0.115, 1.0)
    X, info = wd.bbicggr_solve(ctx, torch.from_numpy(B).cuda(), j=2, tol=1e-12)
    assert info["status"] == wd.WD_OK and abs(info["iters"] - ref.iters) <= 2
    X = X.cpu().numpy()
    assert np.abs(X - ref.X).max() <= 1e-10 * np.abs(ref.X).max()
    wd.wd_destroy(ctx)
