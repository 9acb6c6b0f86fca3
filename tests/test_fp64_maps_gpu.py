"""LENS_FP64 maps against the FP64 oracle around the kernel's chunk of 32
potentials and CTA of 64 nodes, with every kind of potential, circular and
very elliptical ones, and nodes on a potential's axes and centre."""
import numpy as np
import pytest

import oracle
from paper_2004_06352_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
REL = 1e-11  # tolerances.py: LENS_FP64 maps


@pytest.mark.parametrize("n,nx,ny", [(1, 8, 8), (31, 9, 7), (32, 13, 5), (33, 33, 31), (65, 64, 3), (97, 61, 50)])
def test_fp64_maps_match_oracle(lens, n, nx, ny):
    m = I.random_model(n, seed=n, types=(I.DPIE, I.DPIE, I.DPIE, I.SIS, I.POINT), eps_max=0.95)
    m[0, 1:5] = [0.0, 0.0, 0.0, 0.99 if n > 1 else 0.3]   # centred, along the axes, nearly a line
    if n > 2:
        m[1, 4], m[2, 4] = 0.0, 1e-10                     # circular, series
    g = I.grid(nx, field=(-40, 40, -40, 40), ny=ny)
    ref = oracle.maps(m, g, 0.7, 6)
    with lens.Context(0) as ctx:
        mid = ctx.model_upload(m)
        h = torch.empty((6, ny, nx), dtype=torch.float64, device=DEV)
        a = torch.empty((2, ny, nx), dtype=torch.float64, device=DEV)
        ctx.hessian_map(mid, g, 0.7, lens.LENS_FP64, h)
        ctx.grad_map(mid, g, 0.7, lens.LENS_FP64, a)
        ctx.wait()
    for got in (h.cpu().numpy()[:5], a.cpu().numpy()):
        for k in range(len(got)):
            tol = REL * np.maximum(np.abs(ref[k]), 1e-3 * np.abs(ref[k]).max())
            assert np.all(np.abs(got[k] - ref[k]) <= tol), k
