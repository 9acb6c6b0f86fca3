"""Maps streamed to host memory are computed in 1, 3, 6 or 8 row bands by their
size; every value is the device map's (Sec. 4.1 Eq. 10, Sec. 2.4)."""
import pytest
import torch

from paper_2004_06352_gb300 import inputs as I

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# bytes of the output: 1 band up to 8 MiB, 3 up to 128 MiB, then 6; rows that do
# not divide; fewer tile rows than bands; a budget: 8 bands
@pytest.mark.parametrize("nx,ny,hess,prec,budget", [
    (1024, 1024, False, "LENS_MIXED", 0), (1025, 1024, False, "LENS_MIXED", 0), (513, 33, True, "LENS_MIXED", 0),
    (3001, 1900, True, "LENS_MIXED", 0), (4099, 4097, False, "LENS_MIXED", 0), (700, 701, True, "LENS_MIXED", 1 << 30),
    (130, 97, True, "LENS_FP64", 0), (1200, 1203, False, "LENS_FP64", 0)])
def test_banded_host_map_is_the_device_map(lens, nx, ny, hess, prec, budget):
    m = I.cfg2_model(n_members=10 if prec == "LENS_FP64" else 150)
    g = I.grid(nx, field=(-80, 80, -75, 77), ny=ny)
    p, dt, planes = getattr(lens, prec), torch.float64 if prec == "LENS_FP64" else torch.float32, 6 if hess else 2
    with lens.Context(0, mem_budget_bytes=budget) as ctx:
        mid = ctx.model_upload(m)
        dev = torch.full((planes, ny, nx), -1.0, dtype=dt, device=DEV)
        (ctx.hessian_map if hess else ctx.grad_map)(mid, g, 0.7, p, dev)
        ctx.wait()
        for _ in range(2):
            host = torch.full((planes, ny, nx), -2.0, dtype=dt).pin_memory()
            (ctx.hessian_map_host if hess else ctx.grad_map_host)(mid, g, 0.7, p, host)
            ctx.wait()
            assert torch.equal(host, dev.cpu())
