"""Device memory that a context takes (needs a GB300): a solve holds its ten blocks and no copy of an
operand beside them, and the first product on a small lattice allocates nothing."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def random_context(wd, dims):
    V = dims[0] * dims[1] * dims[2] * dims[3]
    g = torch.Generator(device="cuda").manual_seed(1)
    m = 0.2 * torch.view_as_complex(torch.randn((V, 4, 3, 3, 2), generator=g, device="cuda", dtype=torch.float64))
    return wd.wd_create(torch.linalg.qr(torch.eye(3, device="cuda") + m)[0].contiguous(), dims, 0.12, 1.0)


def free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("batch", [False, True])
def test_a_solve_takes_ten_blocks(batch):
    import paper_0907_3261_gb300 as wd
    dims, L = (16, 16, 16, 12), 12
    V = dims[0] * dims[1] * dims[2] * dims[3]
    ctx = random_context(wd, dims)
    B = torch.randn((V, 4, 3, L), dtype=torch.complex128, device="cuda")
    X = torch.zeros_like(B)
    block, before = B.numel() * 16, free()
    if batch:                                            # (one iteration does not converge: no error)
        wd.bbicggr_solve_batch([dict(ctx=ctx, B=B, X=X, j=3, tol=1e-12, maxit=1, max_restarts=0)])
    else:
        wd.bbicggr_solve(ctx, B, X, j=3, tol=1e-12, maxit=1, max_restarts=0)
    assert 10 * block <= before - free() < 10.5 * block
    wd.wd_destroy(ctx)


@pytest.mark.parametrize("dims,L", [((8, 8, 8, 8), 12), ((8, 8, 8, 8), 16), ((12, 12, 12, 24), 1), ((16, 16, 16, 32), 1)])
def test_the_first_small_product_allocates_nothing(dims, L):
    import paper_0907_3261_gb300 as wd
    warm = random_context(wd, (4, 4, 4, 4))              # the kernels' modules are loaded
    wd.wd_apply(warm, torch.ones((256, 4, 3, L), dtype=torch.complex128, device="cuda"))
    V = dims[0] * dims[1] * dims[2] * dims[3]
    ctx = random_context(wd, dims)
    X = torch.randn((V, 4, 3, L), dtype=torch.complex128, device="cuda")
    Y = torch.empty_like(X)
    before = free()
    wd.wd_apply(ctx, X, Y)
    assert free() == before
    wd.wd_destroy(ctx)
    wd.wd_destroy(warm)
