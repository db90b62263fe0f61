"""Halo slices of a domain-decomposed run (needs a GB300): ranks whose FP64 stencils have different forms
exchange one form, and slices whose exponents do not fill 16 bytes keep the callbacks' buffers aligned.
Ranks are processes that share the GPU and exchange on the host, as in test_gpu_domain.py."""
import numpy as np
import pytest

from paper_0907_3261_gb300 import domain as D
from paper_0907_3261_gb300 import inputs as I
from test_gpu_domain import free_port

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DIMS, L, KAPPA, J = (4, 4, 4, 8), 3, 0.12, 4


def worker(rank, world, port, results):
    import os
    import torch.distributed as dist
    os.environ.update(MASTER_ADDR="127.0.0.1", MASTER_PORT=str(port))
    dist.init_process_group("gloo", rank=rank, world_size=world)
    torch.cuda.set_device(0)
    import paper_0907_3261_gb300 as wd
    S = D.slice_sites(DIMS)
    t0, t1 = D.slab_range(DIMS[3], rank, world)
    mine = slice(t0 * S, t1 * S)
    ds = D.DomainSolver(wd, I.random_links(DIMS, 0.2, seed=0)[mine], DIMS, KAPPA, 1.0, dist, rank, world)
    if rank == 1:
        wd.wd_set_apply_form(ds.ctx, 0)
    P = I.gaussian_block(DIMS, L, seed=2)[mine]
    G = ds.interior(wd.jacobi_precond(ds.ctx, ds.extend(P), J)).cpu().numpy()
    X, info = ds.solve(P, j=J, tol=1e-12)
    results[rank] = (G, X.cpu().numpy(), info["status"], info["iters"])
    ds.close()
    dist.barrier()
    dist.destroy_process_group()


def test_ranks_of_different_forms():
    import torch.multiprocessing as mp
    import __graft_entry__
    import paper_0907_3261_gb300 as wd
    from oracle import operator as O
    from oracle import solver as S
    __graft_entry__.build()
    with mp.get_context("spawn").Manager() as m:
        results = m.dict()
        mp.spawn(worker, args=(2, free_port(), results), nprocs=2, join=True)
        res = dict(results)
    links, P = I.random_links(DIMS, 0.2, seed=0), I.gaussian_block(DIMS, L, seed=2)
    ctx = wd.wd_create(torch.from_numpy(links).cuda(), DIMS, KAPPA, 1.0)
    wd.wd_set_apply_form(ctx, 0)
    G = wd.jacobi_precond(ctx, torch.from_numpy(P).cuda(), J).cpu().numpy()
    wd.wd_destroy(ctx)
    assert np.array_equal(np.concatenate([res[0][0], res[1][0]]), G)
    assert res[0][2:] == res[1][2:] and res[0][2] == 0
    op = O.WilsonClover(links, DIMS, KAPPA, 1.0)
    assert S.true_residual(op, P, np.concatenate([res[0][1], res[1][1]])).max() <= 1e-12


@pytest.mark.parametrize("dims,L", [((3, 3, 3, 4), 1), ((3, 5, 3, 3), 3), ((4, 4, 4, 4), 4)])
def test_slices_are_aligned(dims, L):
    import paper_0907_3261_gb300 as wd
    links, P = I.random_links(dims, 0.2, seed=0), I.gaussian_block(dims, L, seed=2)
    ctx = wd.wd_create(torch.from_numpy(links).cuda(), dims, KAPPA, 1.0)
    G = wd.jacobi_precond(ctx, torch.from_numpy(P).cuda(), 5).cpu().numpy()
    wd.wd_destroy(ctx)
    ds = D.DomainSolver(wd, links, dims, KAPPA, 1.0)
    seen = []

    def exchange(*views):
        seen.extend((v.__array_interface__["data"][0] % 16, v.nbytes % 16) for v in views)
        D.exchange_callback()(*views)

    wd.wd_set_domain(ds.ctx, exchange, D.allreduce_callback())
    got = ds.interior(wd.jacobi_precond(ds.ctx, ds.extend(P), 5)).cpu().numpy()
    ds.close()
    assert len(seen) == 16 and set(seen) == {(0, 0)}
    assert np.array_equal(got, G)
