"""Captured products Y = A X (needs a GB300): the graph holds the address of the context's copy of the
operand, which has to outlive a product with more columns on the same context."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,L,larger", [((4, 4, 4, 4), 3, 12), ((16, 16, 16, 12), 3, 12)])
def test_a_captured_product_outlives_a_larger_one(dims, L, larger):
    import paper_0907_3261_gb300 as wd
    V = dims[0] * dims[1] * dims[2] * dims[3]
    g = torch.Generator(device="cuda").manual_seed(1)
    block = lambda n: torch.view_as_complex(torch.randn((V, 4, 3, n, 2), generator=g, device="cuda",
                                                        dtype=torch.float64))
    links, _ = torch.linalg.qr(torch.eye(3, device="cuda") + 0.2 * block(3).reshape(V, 4, 3, 3))
    ctx = wd.wd_create(links.contiguous(), dims, 0.12, 1.0)
    x, y, z = block(L), block(L), block(larger)
    want = wd.wd_apply(ctx, x).clone()
    graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=s):
        wd.wd_apply(ctx, x, y, stream=s)
    first = wd.wd_apply(ctx, z).clone()                  # the copy grows
    # whoever gets freed memory of the copy's size must find it as it was
    torch.cuda.empty_cache()
    own = [torch.zeros(V * 12 * L * 2, dtype=torch.float64, device="cuda") for _ in range(4)]
    y.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, want)
    assert all(not bool(o.any()) for o in own)
    assert torch.equal(wd.wd_apply(ctx, z), first)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, want)
    wd.wd_destroy(ctx)
