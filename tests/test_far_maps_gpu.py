"""LENS_MIXED maps with interpolated far potentials against the FP64 oracle,
at the sizes where the tiles, the node lists and the coarse level end."""
import numpy as np
import pytest

import oracle
from paper_2004_06352_gb300 import inputs as I
from tests import tolerances as T

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# (nx, ny, half-width, model): one node past and one short of 32-node tiles,
# fields much wider and much narrower than the potentials' spread, very
# elliptical terms, more potentials than one staged chunk at a place, no
# cluster-scale potential, only cluster-scale ones
CASES = [
    (513, 479, 60.0, lambda: I.cfg2_model(seed=3, n_members=300)),
    (1025, 33, 60.0, lambda: I.cfg2_model(seed=4, n_members=120)),
    (700, 640, 300.0, lambda: I.cfg2_model(seed=5, n_members=500)),
    (640, 611, 12.0, lambda: I.cfg2_model(seed=6, n_members=900)),
    (961, 767, 60.0, lambda: I.random_model(200, seed=7, types=(I.DPIE, I.DPIE, I.SIS, I.POINT), eps_max=0.9)),
    (1600, 1500, 80.0, lambda: I.member_model(1500, seed=8, field=15.0)),
    (800, 600, 70.0, lambda: I.cfg2_model(seed=9, n_members=0)),
    # most nodes recomputed in double-float, deflection and all planes (dense tiles of the repair)
    (860, 650, 25.0, lambda: I.cfg2_model(seed=12, n_members=700, rcut_star=45.0)),
    (2100, 1900, 25.0, lambda: I.cfg2_model(seed=13, n_members=300, rcut_star=45.0)),
    # few tiles and few potentials; few tiles and several chunks of potentials at a tile's nodes
    (448, 440, 100.0, lambda: I.cfg2_model(seed=14, n_members=8)),
    (385, 383, 60.0, lambda: I.cfg2_model(seed=15, n_members=1100)),
]


def sample(g, rng):
    """Nodes on the tiles' edges and corners and at random."""
    e = np.array([0, 1, 30, 31, 32, 33, 63, 64, 127, 128, 255, 256])
    i = np.concatenate([np.minimum(np.tile(e, len(e)), g["nx"] - 1), [g["nx"] - 1, g["nx"] - 2], rng.integers(0, g["nx"], 3000)])
    j = np.concatenate([np.minimum(np.repeat(e, len(e)), g["ny"] - 1), [g["ny"] - 1, 0], rng.integers(0, g["ny"], 3000)])
    return i, j


@pytest.mark.parametrize("k", range(len(CASES)))
def test_interpolated_maps_match_oracle(lens, k):
    nx, ny, half, make = CASES[k]
    m, g = make(), I.grid(nx, field=(-half, half, -half * 0.9, half * 0.9), ny=ny)
    dx, dy = (g["xmax"] - g["xmin"]) / (nx - 1), (g["ymax"] - g["ymin"]) / (ny - 1)
    i, j = sample(g, np.random.default_rng(k))
    X, Y = g["xmin"] + i * dx, g["ymin"] + j * dy
    ax, ay, hxx, hyy, hxy = oracle.model_eval(m, X, Y, 0.8).T
    ref = (ax, ay, 0.5 * (hxx + hyy), 0.5 * (hxx - hyy), hxy)
    phi_ref = oracle.potential(m, X, Y, 0.8)
    with lens.Context(0) as ctx:
        mid = ctx.model_upload(m)
        h = torch.empty((6, ny, nx), device=DEV)
        a = torch.empty((2, ny, nx), device=DEV)
        phi = torch.empty((1, ny, nx), dtype=torch.float64, device=DEV)
        ctx.hessian_map(mid, g, 0.8, lens.LENS_MIXED, h)
        ctx.grad_map(mid, g, 0.8, lens.LENS_MIXED, a)
        ctx.potential_map(mid, g, 0.8, lens.LENS_MIXED, phi)
        host = torch.empty((6, ny, nx), pin_memory=True)
        ctx.hessian_map_host(mid, g, 0.8, lens.LENS_MIXED, host)
        ctx.wait()
        assert torch.equal(host, h.cpu())
        h, a, phi = h.cpu().numpy()[:, j, i].astype(np.float64), a.cpu().numpy()[:, j, i].astype(np.float64), phi.cpu().numpy()[0, j, i]
    peak = np.hypot(ref[0], ref[1]).max()
    for got in (h[:2], a):
        bad, err, tol = T.alpha_violations(got[0], got[1], ref[0], ref[1], peak=peak)
        assert not bad.any(), (bad.sum(), (err / tol).max())
    assert not T.hess_violations(h[2], h[3], h[4], ref[2], ref[3], ref[4]).any()
    rdet = (1 - ref[2]) ** 2 - ref[3] ** 2 - ref[4] ** 2
    assert not T.mu_violations(h[5], 1 / rdet).any()
    if k not in (4, 7, 8):  # the potential's tolerance is stated for cluster models (members of b0 up to 2.3, r_cut up to 18 arcsec)
        assert np.abs(phi - phi_ref).max() <= T.pot_mixed_tol(phi_ref)


def test_interpolated_map_yields_to_the_budget(lens):
    """A context without room for the coarse level's values still makes the
    map (and the same one within the tolerances)."""
    m, g = I.cfg2_model(seed=10, n_members=400), I.grid(1024)
    out, ref = (torch.empty((2, 1024, 1024), device=DEV) for _ in range(2))
    with lens.Context(0) as ctx:
        mid = ctx.model_upload(m)
        used = ctx.mem_used()
        ctx.grad_map(mid, g, 1.0, lens.LENS_MIXED, ref)
        ctx.wait()
    # 4 bytes per node for the repair list and nothing more
    with lens.Context(0, mem_budget_bytes=used + 4 * 1024 * 1024 + 512) as ctx:
        ctx.grad_map(ctx.model_upload(m), g, 1.0, lens.LENS_MIXED, out)
        ctx.wait()
    o, r = out.cpu().numpy().astype(np.float64), ref.cpu().numpy().astype(np.float64)
    bad, _, _ = T.alpha_violations(o[0], o[1], r[0], r[1], rel=2 * T.ALPHA_REL)
    assert not bad.any()
