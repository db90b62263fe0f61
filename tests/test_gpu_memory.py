"""Device memory that a context takes (needs a GB300): a solve holds its ten blocks and no copy of an
operand beside them, the first product on a small lattice allocates nothing, and a context whose
fixed-point tables find no room runs its products on the FP64 pipe."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def random_links(dims):
    V = dims[0] * dims[1] * dims[2] * dims[3]
    g = torch.Generator(device="cuda").manual_seed(1)
    m = 0.2 * torch.view_as_complex(torch.randn((V, 4, 3, 3, 2), generator=g, device="cuda", dtype=torch.float64))
    m = m + torch.eye(3, device="cuda")
    a = m[..., 0, :] / torch.linalg.vector_norm(m[..., 0, :], dim=-1, keepdim=True)
    b = m[..., 1, :] - (a.conj() * m[..., 1, :]).sum(-1, keepdim=True) * a
    b = b / torch.linalg.vector_norm(b, dim=-1, keepdim=True)
    return torch.stack([a, b, torch.linalg.cross(a, b).conj()], dim=-2).contiguous()


def random_context(wd, dims):
    return wd.wd_create(random_links(dims), dims, 0.12, 1.0)


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


def test_a_context_without_room_for_its_tables():
    """16^3x32: the operator takes 383 MB, the tables 474; 600 MB are left."""
    import paper_0907_3261_gb300 as wd
    dims, L = (16, 16, 16, 32), 1
    warm = random_context(wd, (4, 4, 4, 4))
    wd.wd_apply(warm, torch.ones((256, 4, 3, L), dtype=torch.complex128, device="cuda"))
    links = random_links(dims)
    X = torch.randn((16 ** 3 * 32, 4, 3, L), dtype=torch.complex128, device="cuda")
    full = wd.wd_create(links, dims, 0.12, 1.0)
    wd.wd_set_apply_form(full, 0)
    want = wd.wd_apply(full, X)
    wd.wd_destroy(full)
    Y = torch.zeros_like(X)
    hog = torch.empty(free() - (600 << 20), dtype=torch.uint8, device="cuda")
    try:
        ctx = wd.wd_create(links, dims, 0.12, 1.0)
        assert wd.wd_get_apply_form(ctx) == 0
        with pytest.raises(wd.WDError):
            wd.wd_set_apply_form(ctx, 1)
        wd.wd_apply(ctx, X, Y)
        wd.wd_destroy(ctx)
    finally:
        del hog
        torch.cuda.empty_cache()
    assert torch.equal(Y, want)
    wd.wd_destroy(warm)
