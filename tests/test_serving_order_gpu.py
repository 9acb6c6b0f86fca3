"""The request loop starts the shortest expected work first: a large map whose
far potentials are interpolated before a chi2 batch that takes longer."""
import numpy as np
import pytest

from paper_2004_06352_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_interpolated_map_before_longer_chi2(lens):
    m, cons = I.cfg2_model(), I.random_constraints(100, seed=5, mult=(3, 4))
    n, P = 4096, 150000  # about 3 ms with the copy of 134 MB, and 10 ms
    pars = I.perturbed_params(m, (0, 1), P, seed=6)
    with lens.Context(0) as ctx:
        mid = ctx.model_upload(m)
        cs = ctx.cset_create(mid, cons, (0, 1))
        srv = lens.Server(ctx, slots=1, pool_bytes=1 << 30)
        res = {k: torch.empty(s, dtype=d, pin_memory=True) for k, s, d in
               (("first", P, torch.float64), ("chi2", P, torch.float64), ("map", (2, n, n), torch.float32))}
        tick = {srv.submit_chi2_source(cs, pars, 0, res["first"]): "first"}
        assert srv.progress() == []  # it holds the one slot
        tick[srv.submit_map(mid, I.grid(n), 0.8, lens.LENS_MIXED, False, res["map"])] = "map"
        tick[srv.submit_chi2_source(cs, pars, 0, res["chi2"])] = "chi2"
        order = []
        while len(order) < 3:
            order += [tick[t] for t, status, _, _ in srv.progress() if status == lens.LENS_OK]
        srv.close()
    assert order == ["first", "map", "chi2"]
    assert torch.equal(res["first"], res["chi2"])
