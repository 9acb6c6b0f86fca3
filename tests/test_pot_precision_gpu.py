"""LENS_MIXED potential maps of models whose cluster-scale potentials outweigh
the rest: those are FP64, so the map's error is what the FP32 members leave
(1e-7 of each one's b0 r_cut scale times its logarithm), or nothing, also
where the interpolated form carries them (Sec. 2.1 Eq. 2; Sec. 2.4)."""
import numpy as np
import pytest

import oracle
from paper_2004_06352_gb300 import inputs as I
from tests import tolerances as T

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def tolerance(m, ref):
    """FP64's, and per member 1e-7 of b0 r_cut times the log of D_t ~ (2 r_cut)^2, largest when all agree."""
    s = m[2:, 7] * m[2:, 6] * np.maximum(1.0, np.log(4 * m[2:, 6] ** 2))
    return T.POT_FP64_REL * np.abs(ref).max() + 1e-7 * s.sum()


# 512: 512-thread tiles; 1537: 256 threads, ragged; 4096: 64 x 64 tiles and coarse levels
@pytest.mark.parametrize("n", [512, 1537, 4096])
@pytest.mark.parametrize("members,strength", [(0, 1.0), (8, 0.05), (60, 0.05), (300, 0.05)])
def test_weak_members_potential(lens, n, members, strength):
    m, g = I.cfg2_model(n_members=members), I.grid(n, field=(-60, 60, -60, 60))
    m[2:, 7] *= strength
    with lens.Context(0) as ctx:
        out = torch.empty((2, n, n), dtype=torch.float64, device=DEV)
        ctx.potential_map(ctx.model_upload(m), g, 0.9, lens.LENS_MIXED, out, beta=(0.7, -0.4))
        ctx.wait()
        rng = np.random.default_rng(n)
        i, j = rng.integers(0, n, 12000), rng.integers(0, n, 12000)
        i[:4], j[:4] = [0, n - 1, 0, n - 1], [0, 0, n - 1, n - 1]
        got = out[:, torch.tensor(j, device=DEV), torch.tensor(i, device=DEV)].cpu().numpy()
    x, y = (-60 + k * (120 / (n - 1)) for k in (i, j))
    ref = oracle.potential(m, x, y, 0.9)
    tol = tolerance(m, ref)
    assert np.abs(got[0] - ref).max() <= tol, (np.abs(got[0] - ref).max(), tol)
    tau = 0.5 * ((x - 0.7) ** 2 + (y + 0.4) ** 2) - ref
    assert np.abs(got[1] - tau).max() <= tol


# models that the rule on the members' scales (below 0.0025 of all) leaves to the interpolated form: several
# staged chunks at a tile's nodes with 512 threads, members of large r_cut with 256, a coarse level over a wide field
@pytest.mark.parametrize("n,members,strength,rcut,half", [(385, 1100, 0.3, 8.0, 60.0), (700, 500, 0.2, 45.0, 60.0), (1300, 700, 0.5, 8.0, 300.0)])
def test_interpolated_potential_shapes(lens, n, members, strength, rcut, half):
    m, g = I.cfg2_model(n_members=members, rcut_star=rcut), I.grid(n, field=(-half, half, -half, half), ny=n - 11)
    m[2:, 7] *= strength
    scale = m[:, 7] * m[:, 6]
    assert np.sqrt((scale[2:] ** 2).sum()) <= 0.0025 * scale.sum()
    with lens.Context(0) as ctx:
        out = torch.empty((1, n - 11, n), dtype=torch.float64, device=DEV)
        ctx.potential_map(ctx.model_upload(m), g, 0.9, lens.LENS_MIXED, out)
        ctx.wait()
        rng = np.random.default_rng(n)
        i, j = rng.integers(0, n, 12000), rng.integers(0, n - 11, 12000)
        got = out[0, torch.tensor(j, device=DEV), torch.tensor(i, device=DEV)].cpu().numpy()
    ref = oracle.potential(m, -half + i * (2 * half / (n - 1)), -half + j * (2 * half / (n - 12)), 0.9)
    assert np.abs(got - ref).max() <= min(tolerance(m, ref), T.pot_mixed_tol(ref))
