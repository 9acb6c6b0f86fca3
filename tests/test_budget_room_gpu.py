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
