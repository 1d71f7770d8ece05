"""A batch's launch form follows from its grids, not from the autotuner's clock: a batch with a grid of the line-FFT
passes takes a launch per phase, which is where those passes run (the forms round differently), so that a second
batch of the same problems returns the same bits."""
import numpy as np
import pytest

from paper_1702_04045_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _batch(ecut, nb, precision, nk=1):
    from paper_1702_04045_gb300 import paro
    lat, pos = inputs.diamond_cell(1, 10.26, 91)
    k = [(0.1 * i, 0.0, 0.0) for i in range(nk)]
    ctx = paro.Context(lat, pos, ecut, nb, nb, precision, kpts=k, kweights=np.full(nk, 1 / nk))
    ctx.set_local_pp(**inputs.LOCAL_PP)
    return ctx, paro.Batch([ctx])


@pytest.mark.parametrize("precision,dtype", [("fp64", torch.complex128), ("mixed", torch.complex64)])
@pytest.mark.parametrize("ecut,grid,nb,nk", [(10.0, 32, 1, 1), (10.0, 32, 5, 3), (5.0, 24, 1, 1), (5.0, 24, 5, 3)])
def test_form_follows_from_the_grid(precision, dtype, ecut, grid, nb, nk):
    covered = grid != 24
    outs = []
    for _ in range(2):
        ctx, b = _batch(ecut, nb, precision, nk)
        assert ctx.grid == (grid,) * 3
        forms = set(b.tuning()[:, 0].astype(int))
        assert forms == ({3} if covered else {1, 3})
        psis = [torch.from_numpy(inputs.start_vectors(nb, ctx.npw(ik), ik)).to(dtype).cuda() for ik in range(nk)]
        outs.append(b.apply_h(psis))
        b.close()
    for x, y in zip(*outs):
        assert torch.equal(x, y)
