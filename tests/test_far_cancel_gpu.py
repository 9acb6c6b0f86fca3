"""Interpolated LENS_MIXED maps where the deflections of cluster-scale
potentials cancel: next to the zero of alpha the rounding of the interpolated
remainders, which no FP32 potential's magnitude stands for, is larger than
1e-6 |alpha|, so those nodes have to be recomputed in double-float whatever
the members' strength, also where there are none.  Checked against the FP64
oracle on the nodes of smallest deflection (Sec. 4.1 Eq. 10; Sec. 2.4)."""
import numpy as np
import pytest

import oracle
from paper_2004_06352_gb300 import inputs as I
from tests import tolerances as T

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def pair(d, members=0):
    """Two b0 = 30" clusters at (+-d, 0) and weak members between them."""
    rows = [I.halo_row(I.DPIE, s * d, 0.0, 0.4 * s, 0.25, 4.0, 900.0, 30.0) for s in (-1.0, 1.0)]
    rng = np.random.default_rng(members)
    for _ in range(members):
        x0, y0 = rng.uniform(-60, 60, 2)
        rows.append(I.halo_row(I.DPIE, x0, y0, 0.3, 0.2, 0.05, 4.0, 0.1))
    return np.stack(rows)


CASES = [  # model, nodes a side, hessian
    (lambda: pair(40.0, 8), 2048, True), (lambda: pair(40.0, 60), 2048, False), (lambda: pair(40.0, 8), 4096, False),
    (lambda: pair(90.0), 2048, True), (lambda: pair(60.0), 512, True), (lambda: pair(60.0), 512, False),
    (lambda: I.cfg2_model(seed=8, n_members=0), 4096, True), (lambda: I.cfg2_model(seed=4, n_members=8), 1024, True)]


# (with the repair of the FP32 terms off: the models without any)
@pytest.mark.parametrize("k,ratio", [(k, None) for k in range(len(CASES))] + [(k, 0.0) for k in (3, 4, 5, 6)])
def test_zero_of_cluster_deflection(lens, k, ratio):
    make, n, hess = CASES[k]
    m, g = make(), I.grid(n)
    with lens.Context(0) as ctx:
        if ratio is not None:
            ctx.set_repair_ratio(ratio)
        mid = ctx.model_upload(m)
        out = torch.empty((6 if hess else 2, n, n), device=DEV)
        (ctx.hessian_map if hess else ctx.grad_map)(mid, g, 0.8, lens.LENS_MIXED, out)
        host = torch.empty(out.shape, pin_memory=True)
        (ctx.hessian_map_host if hess else ctx.grad_map_host)(mid, g, 0.8, lens.LENS_MIXED, host)
        ctx.wait()
        assert torch.equal(host, out.cpu())
        a = torch.hypot(out[0], out[1])
        peak = float(a.max())
        idx = torch.topk(a.ravel(), 40000, largest=False).indices
        j, i = (idx // n).cpu().numpy(), (idx % n).cpu().numpy()
        got = out[:, idx // n, idx % n].cpu().numpy().astype(np.float64)
    step = 200.0 / (n - 1)
    ax, ay, hxx, hyy, hxy = oracle.model_eval(m, -100.0 + i * step, -100.0 + j * step, 0.8).T
    bad, err, tol = T.alpha_violations(got[0], got[1], ax, ay, peak=peak)
    assert not bad.any(), (bad.sum(), (err / tol).max())
    if hess:
        ka, g1 = 0.5 * (hxx + hyy), 0.5 * (hxx - hyy)
        assert not T.hess_violations(got[2], got[3], got[4], ka, g1, hxy).any()
        assert not T.mu_violations(got[5], 1 / ((1 - ka) ** 2 - g1 ** 2 - hxy ** 2)).any()
