"""Reciprocal, reciprocal square root and square root of the LENS_FP64 maps
(one third-order step on the MUFU seed) against IEEE division and square root,
over positive normal doubles from 1e-300 to 1e300."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_third_order_steps_within_two_ulp(lens):
    """1 ulp for the reciprocal (one rounding of a correction below 2^-52 of
    it), 2 for the roots (the rounding of a y^2 halved, and the last one)."""
    rng = np.random.default_rng(4)
    x = np.concatenate([10.0 ** rng.uniform(-300, 300, 40000), rng.uniform(0.5, 4.0, 40000),
                        [1.0, 2.0, 0.5, 3.0, 4.0, 1e-300, 1e300, np.nextafter(1.0, 2.0), np.nextafter(2.0, 0.0), np.nextafter(4.0, 0.0)]])
    with lens.Context(0) as ctx:
        out = torch.empty((3, x.size), dtype=torch.float64, device=DEV)
        ctx.selftest_math_maps(torch.tensor(x, device=DEV), out)
        ctx.wait()
        rcp, rs, sq = out.cpu().numpy()
    ulps = lambda a, b: (np.abs(a - b) / np.spacing(b)).max()
    assert ulps(rcp, 1.0 / x) <= 1.0
    assert ulps(rs, (np.longdouble(1) / np.sqrt(x.astype(np.longdouble))).astype(np.float64)) <= 2.0
    assert ulps(sq, np.sqrt(x)) <= 2.0
