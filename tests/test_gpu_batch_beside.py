"""Batches that live beside each other: the kernels' shared-memory limit is that of the largest, whichever was created
last. Planes of 96 x 96 points need 73 KB a CTA in FP32, units of 24 x 24 points at most half of it."""
import numpy as np
import pytest

from paper_1702_04045_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("first,second", [(96, 24), (24, 96)])
def test_an_older_batch_keeps_working(first, second):
    from paper_1702_04045_gb300 import paro

    def batch(n):
        # a flat cell: n x n planes, few of them, which the line FFTs (cubic grids) leave to the shared-memory passes
        lat = np.diag([n / 1.4, n / 1.4, 7.0])
        pos = np.random.default_rng(n).uniform(0, 1, (2, 3)) @ lat
        ctx = paro.Context(lat, pos, 2.0, 4, 4, "mixed")
        ctx.set_local_pp(**inputs.LOCAL_PP)
        x = inputs.start_vectors(4, ctx.npw(), 5)
        ctx.set_orbitals(x)
        x = torch.from_numpy(x.astype(np.complex64)).cuda()
        return ctx, paro.Batch([ctx]), x

    a, b = batch(first), batch(second)
    assert a[0].grid == (first, first, 9) and b[0].grid == (second, second, 9)
    for ctx, bt, x in (a, b, a):
        assert torch.equal(bt.apply_h([x])[0], bt.apply_h([x])[0])
        ref = ctx.apply_h(x)
        assert float((bt.apply_h([x])[0] - ref).abs().max()) < 2e-6 * float(ref.abs().max())
        bt.step(0.25, 2)
