"""Cholesky orthonormalisation of more rows than 64 blocks of one cluster's order (192 rows at most): the blocks' breakdown
flags are as many as the order needs."""
import numpy as np
import pytest

from paper_1702_04045_gb300 import inputs, paro

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_orthonormalisation_of_many_rows():
    n = 12300  # above 64 x 192
    lat, pos = inputs.diamond_cell(2, 10.26, 91)
    ctx = paro.Context(lat, pos, 15.0, 4, 4, "fp64")
    ctx.set_local_pp(**inputs.LOCAL_PP)
    npw = ctx.npw()
    assert npw > 1.9 * n
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.complex(*(torch.randn((n, npw), generator=g, device="cuda", dtype=torch.float64) for _ in range(2)))
    y = ctx.orthonormalize(x)
    rows = torch.linspace(0, n - 1, 96).long().cuda()
    gram = y[rows].conj() @ y.T
    gram[torch.arange(96), rows] -= 1
    # random rows: kappa(S) = ((1 + q)/(1 - q))^2, q = sqrt(n / npw) = 0.72, below 40; n eps kappa
    assert float(gram.abs().max()) < 4 * n * 2.0 ** -52 * 40
    # row i is a combination of the rows up to i: orthogonal to what the rows before it span
    i = int(rows[40])
    assert float((x[:i].conj() @ y[i]).abs().max()) < 4 * n * 2.0 ** -52 * 40 * float(npw) ** 0.5
    del x, y, gram
    torch.cuda.empty_cache()
