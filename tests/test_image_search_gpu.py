"""The image search leaves out blocks of 8 x 8 grid cells that its bound says
hold no image; it must lose none: checked against the oracle's search of every
cell (Sec. 2.3, Fig. 4) on grids with whole and ragged blocks, under varying
potentials of every kind."""
import numpy as np
import pytest
import torch

import oracle
from paper_2004_06352_gb300 import inputs as I
from tests.test_chi2_image_gpu import gpu_images

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# 128 cells: one CTA's columns; 129, 137: blocks of one cell; 250 x 91: ragged both ways
@pytest.mark.parametrize("nx,ny", [(129, 129), (130, 202), (138, 130), (251, 92)])
@pytest.mark.parametrize("kind", ["dpie", "sis", "point"])
def test_no_image_lost(lens, nx, ny, kind):
    """Every well-conditioned oracle image (difficulty < 100) is found within
    1e-6", and every image found is a root to 1e-9": the bounds of the other
    image searches' parity checks."""
    second = {"dpie": I.halo_row(I.DPIE, -12.0, 7.0, 1.1, 0.6, 3.0, 500.0, 11.0),
              "sis": I.halo_row(I.SIS, -12.0, 7.0, 0.0, 0.0, 0.0, 0.0, 9.0),
              "point": I.halo_row(I.POINT, -12.0, 7.0, 0.0, 0.0, 0.0, 0.0, 6.0)}[kind]
    m = np.vstack([I.halo_row(I.DPIE, 0.5, -0.3, 0.4, 0.45, 5.0, 900.0, 25.0), second,
                   I.member_model(8, seed=45, field=45)])
    cons = I.random_constraints(24, seed=86, mult=(2, 2), field=40)
    g = I.grid(nx, field=(-60, 60, -55, 58), ny=ny)
    params = I.perturbed_params(m, (0, 1), 2, seed=nx)
    with lens.Context(0) as ctx:
        cs = ctx.cset_create(ctx.model_upload(m), cons, (0, 1))
        imgs = gpu_images(ctx, cs, g, params)
    seen = 0
    for p in range(2):
        mp = oracle.apply_params(m, (0, 1), params[p])
        _, bary = oracle.backtrace(mp, cons)
        ag = oracle.alpha_grid(mp, g)
        for i, r in enumerate(cons["dls_ds"]):
            ref, _, dif = oracle.find_images(mp, g, r, bary[i], ag=ag, with_difficulty=True)
            mine = imgs[p][imgs[p][:, 2] == i, :2]
            for x, d in zip(ref, dif):
                hit = len(mine) > 0 and np.min(np.hypot(*(mine - x).T)) < 1e-6
                assert hit or d >= 100, (p, i, x, d)
                seen += hit
            for y in mine:
                ev = oracle.model_eval(mp, y[0], y[1], r)[0]
                assert np.hypot(*(y - ev[:2] - bary[i])) < 1e-9, (p, i, y)
    assert seen >= 48
