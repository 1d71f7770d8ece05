"""Row updates of the FP64 iteration (csrc/k_linalg.cu, k_gemm_wx) at the edges of their tiles: the Cholesky factor
and the Rayleigh-Ritz rotation of n rows must leave their span and make them orthonormal."""
import numpy as np
import pytest
import torch

from paper_1702_04045_gb300 import inputs, paro

pytestmark = pytest.mark.gpu


# one row, both sides of the 32-row tile, tiles of 48 rows (33..48, 129..144) and the sizes next to them
@pytest.mark.parametrize("n", [1, 32, 33, 48, 49, 64, 129, 144, 145])
def test_rows_keep_their_span_and_become_orthonormal(n):
    lat, pos = inputs.diamond_cell(1, 10.26, 91)
    ctx = paro.Context(lat, pos, 12.0, n, min(n, 4), "fp64")
    ctx.set_veff(np.zeros(ctx.grid))
    psi = inputs.start_vectors(n, ctx.npw(), n)
    ctx.set_orbitals(torch.from_numpy(psi).cuda())
    out = ctx.get_orbitals()
    # random rows, npw >= 4 n: condition number kappa < 10, sums of up to n terms rounded to 2^-53 of their norms in
    # the Gram matrix, the factor, the update and the rotation: 4 n kappa eps
    tol = 40 * max(n, 8) * 2.0 ** -52
    assert ctx.npw() >= 4 * n
    assert np.abs(out.conj() @ out.T - np.eye(n)).max() <= tol
    left = psi - (psi @ out.conj().T) @ out
    assert (np.linalg.norm(left, axis=1) <= tol * np.linalg.norm(psi, axis=1)).all()
