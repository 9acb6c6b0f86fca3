"""Contexts with a memory budget (include/lens.h): calls that fit before the
optional working memory of the faster forms still run, and as much of that
memory as fits is used."""
import numpy as np
import pytest

from paper_2004_06352_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def uploaded(lens, m):
    with lens.Context(0) as ctx:
        ctx.model_upload(m)
        return ctx.mem_used()


def test_streamed_map_in_small_bands(lens):
    """Eight bands of whole tiles of the direct kernel and one band's list."""
    m, nx, ny = I.cfg2_model(n_members=8), 8192, 256  # (64 x 64 tiles)
    g = I.grid(nx, field=(-50, 50, -1.56, 1.56), ny=ny)
    host, dev = torch.empty((2, ny, nx), pin_memory=True), torch.empty((2, ny, nx), device=DEV)
    rows = 32
    budget = uploaded(lens, m) + 2 * (2 * 4 * rows * nx) + 4 * rows * nx + 4096
    with lens.Context(0, mem_budget_bytes=budget) as ctx:
        ctx.grad_map_host(ctx.model_upload(m), g, 0.8, lens.LENS_MIXED, host)
        ctx.wait()
    with lens.Context(0) as ctx:
        ctx.grad_map(ctx.model_upload(m), g, 0.8, lens.LENS_MIXED, dev)
        ctx.wait()
    dev = dev.cpu()
    assert float((host - dev).abs().max()) <= 2e-6 * float(dev.abs().max())


@pytest.mark.parametrize("host", [False, True])
def test_interpolated_without_dense_repair(lens, host):
    """Room for the coarse level but not for the dense repair's arrays: still
    the interpolated form (the same bits but at repaired nodes)."""
    m, g = I.cfg2_model(seed=10, n_members=400), I.grid(1024)
    out, ref = torch.empty((2, 1024, 1024), pin_memory=True), torch.empty((2, 1024, 1024), device=DEV)
    used = uploaded(lens, m)
    with lens.Context(0) as ctx:
        ctx.grad_map(ctx.model_upload(m), g, 1.0, lens.LENS_MIXED, ref)
        ctx.wait()
    room = (2 << 20) + (2 * 8 * 128 * 1024 + 4 * 128 * 1024 if host else 4 * 1024 * 1024) + 4096
    with lens.Context(0, mem_budget_bytes=used + room) as ctx:
        mid = ctx.model_upload(m)
        if host:
            ctx.grad_map_host(mid, g, 1.0, lens.LENS_MIXED, out)
        else:
            d = torch.empty((2, 1024, 1024), device=DEV)
            ctx.grad_map(mid, g, 1.0, lens.LENS_MIXED, d)
            out = d
        ctx.wait()
    same = (out.cpu() == ref.cpu()).double().mean()
    assert same > 0.99, float(same)


def test_image_search_keeps_the_grid_alone(lens):
    """Under a budget the search's model of a grid is working memory: a grid
    costs its 8 bytes per node, and the results are the same."""
    m, cons = I.cfg2_model(n_members=40), I.random_constraints(8, seed=9, field=30)
    g, P = I.grid(500), 3
    p = torch.tensor(I.perturbed_params(m, (0, 1), P, seed=2), device=DEV)
    res = []
    for budget in (0, 1 << 30):
        with lens.Context(0, mem_budget_bytes=budget) as ctx:
            cs = ctx.cset_create(ctx.model_upload(m), cons, (0, 1))
            chi2, found = torch.empty(P, dtype=torch.float64, device=DEV), torch.empty((P, 8), dtype=torch.int32, device=DEV)
            used = ctx.mem_used()
            ctx.chi2_image(cs, g, p, P, chi2, found)
            ctx.wait()
            kept = ctx.mem_used() - used
            if budget:
                assert kept <= 8 * 500 * 500 + 256, kept
                srv = lens.Server(ctx, slots=1, pool_bytes=64 << 20)
                r = torch.empty(P, dtype=torch.float64, pin_memory=True)
                srv.submit_chi2_image(cs, g, p.cpu().numpy(), r)
                while not srv.progress():
                    pass
                srv.close()
                assert torch.equal(r, chi2.cpu())
            res.append((chi2.cpu(), found.cpu()))
    assert torch.equal(res[0][0], res[1][0]) and torch.equal(res[0][1], res[1][1])
