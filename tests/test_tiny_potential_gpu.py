"""A cluster-scale potential of tiny size at nodes inside it: its denominators
leave the range of the double-float evaluator, which has to hand it to the
FP64 one (Sec. 2.1; Elliptical dPIE of Sec. 2.2)."""
import numpy as np
import pytest

from paper_2004_06352_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("scale", [1e-11, 2e-14, 1e-15, 1e-17])
def test_tiny_cluster_potential(lens, scale):
    m = np.stack([I.halo_row(I.DPIE, 0.0, 0.0, 0.4, 0.3, scale, 3 * scale, 30.0),
                  I.halo_row(I.DPIE, 40.0, -30.0, 0.2, 0.2, 0.2, 20.0, 1.0)])
    g = I.grid(33, field=(-5 * scale, 5 * scale, -5 * scale, 4 * scale), ny=31)
    with lens.Context(0) as ctx:
        ctx.set_repair_ratio(0.0)
        mid = ctx.model_upload(m)
        mixed, plain = torch.empty((2, 31, 33), device=DEV), torch.empty((2, 31, 33), dtype=torch.float64, device=DEV)
        ctx.grad_map(mid, g, 0.8, lens.LENS_MIXED, mixed)
        ctx.grad_map(mid, g, 0.8, lens.LENS_FP64, plain)
        ctx.wait()
    e = torch.hypot(*(mixed.double() - plain))
    assert bool((e <= 1e-6 * torch.hypot(*plain).max()).all()), float(e.max())
