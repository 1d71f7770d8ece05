"""Adjoints of two contexts on two host threads: the long grid's local part needs 166 KB of shared memory a CTA, the
short one's 12 KB, and neither call may see the other's limit."""
import math
import threading

import numpy as np
import pytest

from paper_1702_04045_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_contexts_with_short_and_long_grids_on_two_threads():
    from paper_1702_04045_gb300 import paro
    jobs = []
    for n3 in (324, 24):
        lat = np.diag([6.0, 7.0, (n3 - 4) * math.pi / 4.0])
        ctx = paro.Context(lat, np.random.default_rng(n3).uniform(0, 1, (3, 3)) @ lat, 2.0, 2, 2, "mixed")
        ctx.set_local_pp(**inputs.LOCAL_PP)
        x = torch.from_numpy(inputs.start_vectors(2, ctx.npw(), 6).astype(np.complex64)).cuda()
        ref = ctx.apply_h_adjoint(x, x, grads=("pos",))[2].cpu()
        jobs.append((ctx, x, ref, []))

    def loop(ctx, x, ref, errors):
        try:
            for _ in range(400):
                got = ctx.apply_h_adjoint(x, x, grads=("pos",))[2]
            if not torch.equal(got.cpu(), ref):
                errors.append("values")
        except paro.ParoError as e:
            errors.append(str(e))

    threads = [threading.Thread(target=loop, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert [j[3] for j in jobs] == [[], []]
