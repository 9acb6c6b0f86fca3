"""Source-plane chi2 launch shapes (threads per (image, potential) or image
pairs) against the FP64 oracle at the edges of their rules: odd image counts
and a lone last image, one image, SIS and point-mass varying potentials, more
images than a CTA keeps positions for; and the Metropolis step's copies at
chain counts around a warp."""
import numpy as np
import pytest

import oracle
from paper_2004_06352_gb300 import inputs as I
from tests import tolerances as T

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def constraints(nimg, seed):
    """nimg images: sources of 3, the last with the rest."""
    off = np.append(np.arange(0, max(nimg - 2, 1), 3), nimg)
    rng = np.random.default_rng(seed)
    n = len(off) - 1
    return I.constraints_dict(off, rng.uniform(-40, 40, nimg), rng.uniform(-40, 40, nimg), np.full(nimg, 0.1),
                              rng.uniform(0.5, 0.9, n))


@pytest.mark.parametrize("P,nimg", [(3, 1), (40, 64), (40, 65), (152, 129), (153, 161), (200, 37), (1217, 139), (1300, 203), (9, 2300)])
@pytest.mark.parametrize("var", [(0, 1), (3, 4)])
def test_launch_shapes_match_oracle(lens, P, nimg, var):
    m = I.random_model(30, seed=nimg, types=(I.DPIE, I.DPIE, I.DPIE, I.SIS, I.POINT), field=35)
    cons = constraints(nimg, P)
    params = I.perturbed_params(m, var, P, seed=5)
    for k in range(2):  # SIS and point masses carry no shape
        params[:, 7 * k + 4:7 * k + 6] = np.maximum(params[:, 7 * k + 4:7 * k + 6], [0.01, 0.02])
    n = min(P, 12)
    with lens.Context(0) as ctx:
        cs = ctx.cset_create(ctx.model_upload(m), cons, var)
        d = torch.tensor(params, device=DEV)
        out = torch.empty(P, dtype=torch.float64, device=DEV)
        for variant in (2, 0):
            ctx.chi2_source(cs, d, P, variant, out)
            ctx.wait()
            got = out.cpu().numpy()
            pick = np.r_[0:n - 2, P - 2:P] if P > n else np.arange(P)
            ref = oracle.chi2_source_batch(m, cons, var, params[pick], variant)
            assert np.all(np.abs(got[pick] - ref) <= T.CHI2_REL * np.abs(ref) + 1e-12), variant


@pytest.mark.parametrize("W", [1, 31, 33, 97])
def test_metropolis_copies_match_oracle(lens, W):
    m, cons = I.cfg2_model(seed=11, n_members=20), I.random_constraints(9, seed=12, field=30)
    p0 = I.perturbed_params(m, (0, 1), W, seed=13)
    c0 = oracle.chi2_source_batch(m, cons, (0, 1), p0, 0)
    sig = np.tile([0.1, 0.1, 0.01, 0.02, 0.01, 1.0, 0.05], 2)
    with lens.Context(0) as ctx:
        cs = ctx.cset_create(ctx.model_upload(m), cons, (0, 1))
        p, c = torch.tensor(p0, device=DEV), torch.tensor(c0, device=DEV)
        acc = torch.empty(W, dtype=torch.int32, device=DEV)
        ctx.mcmc_step(cs, p, c, W, torch.tensor(sig, device=DEV), 1e3, 3, 4, torch.empty(16 * W, dtype=torch.float64, device=DEV), acc)
        ctx.wait()
        p, acc = p.cpu().numpy(), acc.cpu().numpy()
    ref = oracle.mcmc_step(m, cons, (0, 1), p0, c0, sig, 1e3, 3, 4)[0]
    assert np.array_equal(acc.astype(bool), (ref != p0).any(axis=1))
    assert np.abs(p - ref).max() <= 1e-12
