"""Eigensolves of two contexts on two host threads: a large and a small order share the solver's kernels, whose
shared-memory limit must not follow the call that set it last."""
import threading

import numpy as np
import pytest

from paper_1702_04045_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_large_and_small_orders_on_two_threads(precision):
    from paper_1702_04045_gb300 import paro
    lat, pos = inputs.diamond_cell(1, 10.26, 91)
    jobs = []
    for n, reps in ((144, 60), (12, 400)):
        ctx = paro.Context(lat, pos, 5.0, 4, 4, precision)
        rng = np.random.default_rng(n)
        a = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
        a = torch.from_numpy(a + a.conj().T).cuda()
        jobs.append((ctx, a, ctx.eigh(a)[0].cpu(), reps, []))

    def loop(ctx, a, ref, reps, errors):
        try:
            for _ in range(reps):
                w = ctx.eigh(a)[0]
            if float((w.cpu() - ref).abs().max()) > 1e-10:
                errors.append("values")
        except paro.ParoError as e:
            errors.append(str(e))

    threads = [threading.Thread(target=loop, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert [j[4] for j in jobs] == [[], []]
