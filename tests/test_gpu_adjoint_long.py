"""Position gradient on elongated cells (non-cubic grids) against the FP64 oracle. The local part stages 32 columns of
the grid along N3 in shared memory, a warp per atom: odd and even N3 up to 324, the longest that the transform of
the local pseudopotential takes (the next is 384), with one atom more than the warps of a CTA."""
import math

import numpy as np
import pytest

from oracle import adjoint, pw
from paper_1702_04045_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n3", [24, 128, 243, 324])
def test_position_gradient_on_long_grids(n3):
    from paper_1702_04045_gb300 import paro
    ecut, nb = 2.0, 3
    # the density sphere reaches 2 |a3| / pi along a3 and the wavefunctions span as much; no G on either sphere itself
    lat = np.diag([6.0, 7.0, (n3 - 3.3) * math.pi / 4.0])
    rng = np.random.default_rng(n3)
    pos = rng.uniform(0, 1, (9, 3)) @ lat
    d = inputs.kb_strengths(len(pos), 5)
    ctx = paro.Context(lat, pos, ecut, nb, nb, "mixed")
    ctx.set_local_pp(**inputs.LOCAL_PP)
    ctx.set_kb(inputs.KB_RC, d)
    assert ctx.grid[2] == n3 and ctx.grid[0] != ctx.grid[2]
    b = pw.Basis(lat, ecut, ctx.grid)
    assert b.npw == ctx.npw()
    psi, w = (inputs.start_vectors(nb, b.npw, s).astype(np.complex64) for s in (6, 7))
    _, _, g = ctx.apply_h_adjoint(torch.from_numpy(psi).cuda(), torch.from_numpy(w).cuda(), grads=("pos",))
    p64, w64 = psi.astype(np.complex128), w.astype(np.complex128)
    ref = (adjoint.grad_pos_local(b, pos, inputs.LOCAL_PP, adjoint.grad_v(b, p64, w64))
           + adjoint.grad_pos_kb(b, pos, (inputs.KB_RC, d), p64, w64))
    # FP32 transforms and 3xTF32 projections: the bound of the adjoint's other FP32 tests
    assert np.abs(g.cpu().numpy() - ref).max() < 2e-5 * np.abs(ref).max()
