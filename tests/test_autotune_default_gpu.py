"""The source-plane chi2's autotuner against the rule it replaces: the shape it
keeps is never slower than the untuned call (Sec. 2.2, Eq. 4)."""
import numpy as np
import pytest

from paper_2004_06352_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# one thread per (image, potential) by default: few images, a set per SM
@pytest.mark.parametrize("P,nsrc", [(4096, 12), (100, 90), (4096, 90)])
def test_tuned_is_not_slower(lens, P, nsrc):
    m, cons = I.cfg2_model(n_members=20), I.random_constraints(nsrc, seed=3, mult=(3, 4))
    with lens.Context(0) as ctx:
        cs = ctx.cset_create(ctx.model_upload(m), cons, (0, 1))
        p = torch.tensor(I.perturbed_params(m, (0, 1), P, seed=4), device=DEV)
        out, ref = torch.empty(P, dtype=torch.float64, device=DEV), torch.empty(P, dtype=torch.float64, device=DEV)

        def best():
            t = []
            for _ in range(30):
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                a.record()
                for _ in range(10):
                    ctx.chi2_source(cs, p, P, 0, out)
                b.record()
                b.synchronize()
                t.append(a.elapsed_time(b))
            return min(t)

        before = best()
        ref.copy_(out)
        ctx.chi2_autotune(cs, p, P, out)
        after = best()
        assert torch.allclose(out, ref, rtol=1e-12, atol=0)
    assert after <= 1.1 * before, (after, before)
