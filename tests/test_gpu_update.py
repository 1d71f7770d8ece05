"""Dense products of csrc/k_linalg.cu at the edges of their tiles. Row updates of the FP64 iteration (k_gemm_wx): the Cholesky factor
and the Rayleigh-Ritz rotation of n rows must leave their span and make them orthonormal."""
import numpy as np
import pytest
import torch

from oracle import pw
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


# FP32 projector products on the CUDA cores: one row, both sides of the 32-row and 64-row update tiles; 4 Ha leaves a
# few K slices, 14 Ha more than the eight lanes of the reduction
@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 65])
@pytest.mark.parametrize("ecut", [4.0, 14.0])
def test_small_fp32_projector_products(n, ecut):
    lat, pos = inputs.diamond_cell(1, 10.26, 91)
    ctx = paro.Context(lat, pos, ecut, 4, 4, "mixed")
    ctx.set_local_pp(**inputs.LOCAL_PP)
    d = inputs.kb_strengths(len(pos), 92)
    ctx.set_kb(inputs.KB_RC, d)
    b = pw.Basis(lat, ecut, ctx.grid)
    beta = pw.kb_beta(lat, pos, b.q, inputs.KB_RC)
    psi = (inputs.start_vectors(n, b.npw, n) * 10.0 ** np.random.default_rng(n).uniform(-6, 6, (n, 1))).astype(np.complex64)
    got = ctx.apply_vnl(torch.from_numpy(psi).cuda()).cpu().numpy()
    ref = (pw.kb_dvec(d)[:, None] * (beta.conj() @ psi.astype(np.complex128).T)).T @ beta
    # FP32 operands, sums of 16 products, then of the 32 projectors: 64 roundings to 2^-24 of the rows' norms
    bound = 64 * 2.0 ** -24 * np.abs(pw.kb_dvec(d)).max() * np.linalg.norm(beta) ** 2
    assert (np.linalg.norm(got - ref, axis=1) <= bound * np.linalg.norm(psi.astype(np.complex128), axis=1)).all()
