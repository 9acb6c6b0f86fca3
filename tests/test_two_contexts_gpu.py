"""Contexts on one device, one host thread each (include/lens.h): the launches
of small and of very large models, which need different amounts of shared
memory, do not disturb each other."""
import threading

import pytest

from paper_2004_06352_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_small_and_large_models_in_threads(lens):
    g = I.grid(512)  # (the same kernels for both models)
    small, large = I.cfg2_model(seed=1, n_members=98), I.cfg2_model(seed=2, n_members=15998)
    errors, same, done = [], [], threading.Event()

    def loop(m, calls):
        try:
            st = torch.cuda.Stream()
            out, ref = (torch.empty((6, 512, 512), device=DEV) for _ in range(2))
            with lens.Context(0) as ctx:
                mid = ctx.model_upload(m)
                r = 0
                while r < calls or (calls == 0 and not done.is_set()):
                    ctx.hessian_map(mid, g, 0.8, lens.LENS_MIXED, out if r else ref, stream=st)
                    r += 1
                    if r % 8 == 0:
                        ctx.wait(st)
                ctx.wait(st)
                same.append(torch.equal(out, ref))
        except Exception as e:
            errors.append(str(e))
        finally:
            if calls:
                done.set()

    t = [threading.Thread(target=loop, args=a) for a in ((large, 80), (small, 0), (small, 0), (small, 0))]
    for x in t:
        x.start()
    for x in t:
        x.join()
    assert not errors and all(same), (errors, same)
