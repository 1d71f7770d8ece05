"""Digit-sliced FP64 products (csrc/k_slice.cu) at the edges of their tiles: Gram, Cholesky apply and the
Kleinman-Bylander products of FP64 rows against extended precision."""
import numpy as np
import pytest
import torch

from oracle import pw
from paper_1702_04045_gb300 import inputs, paro

pytestmark = pytest.mark.gpu


def _ctx(ecut=5.0, kb=True):
    lat, pos = inputs.diamond_cell(1, 10.26, 91)
    ctx = paro.Context(lat, pos, ecut, 4, 4, "fp64")
    ctx.set_local_pp(**inputs.LOCAL_PP)
    d = inputs.kb_strengths(len(pos), 92)
    if kb:
        ctx.set_kb(inputs.KB_RC, d)
    return ctx, lat, pos, d


# Products of n rows: one row, both sides of the 32-column tile, both sides of the 128-row tile
@pytest.mark.parametrize("n", [1, 31, 32, 33, 127, 128, 129, 160])
def test_vnl_against_extended_precision(n):
    ctx, lat, pos, d = _ctx()
    b = pw.Basis(lat, 5.0, ctx.grid)
    beta = pw.kb_beta(lat, pos, b.q, inputs.KB_RC).astype(np.clongdouble)
    rng = np.random.default_rng(n)
    psi = inputs.start_vectors(n, b.npw, n) * 10.0 ** rng.uniform(-12, 6, size=(n, 1))
    got = ctx.apply_vnl(torch.from_numpy(psi).cuda()).cpu().numpy()
    proj = np.conj(beta) @ psi.astype(np.clongdouble).T
    ref = (pw.kb_dvec(d)[:, None] * proj).T @ beta
    # two products, operands and sums rounded to 2^-53 of their rows' norms, and the table of the library
    # against the oracle's (1e-15 relative): 8 eps of ||D|| ||beta||^2 ||psi||
    err = np.linalg.norm((got - ref).astype(np.complex128), axis=1)
    bound = 8 * 2.0 ** -52 * np.abs(d).max() * float(np.linalg.norm(beta.astype(np.complex128), 2)) ** 2
    assert (err <= bound * np.linalg.norm(psi, axis=1)).all()


@pytest.mark.parametrize("n", [2, 32, 33, 130])
def test_rows_of_uneven_size_are_orthonormalised_alike(n):
    """Scaling the rows by powers of two scales every step of the orthonormalisation exactly, so the result
    must not change in a single bit: no row loses digits to a larger one."""
    ctx, _, _, _ = _ctx(kb=False)
    x = torch.from_numpy(inputs.start_vectors(n, ctx.npw(), 7)).cuda()
    s = 2.0 ** np.random.default_rng(n).integers(-60, 60, size=(n, 1)).astype(np.float64)
    a, b = ctx.orthonormalize(x), ctx.orthonormalize(x * torch.from_numpy(s).cuda())
    assert torch.equal(a, b)
    gram = (a.conj() @ a.T).cpu().numpy()
    assert np.abs(gram - np.eye(n)).max() < 1e-13


def test_nonfinite_rows_stay_visible():
    ctx, _, _, _ = _ctx()
    x = torch.from_numpy(inputs.start_vectors(3, ctx.npw(), 7)).cuda()
    x[1, 5] = complex(float("nan"), 0.0)
    out = ctx.apply_vnl(x)
    assert torch.isnan(torch.view_as_real(out[1])).all()
    assert torch.isfinite(torch.view_as_real(out[[0, 2]])).all()
    with pytest.raises(paro.ParoError):
        ctx.orthonormalize(x)


# orders around the blocked cluster kernel's limit and above it: 2 x 2 blocks, then blocks of blocks
@pytest.mark.parametrize("n", [175, 193, 208, 300, 401])
def test_orthonormalisation_by_blocks(n):
    ctx, _, _, _ = _ctx(ecut=8.0, kb=False)
    x = inputs.start_vectors(n, ctx.npw(), n) + 0.3 * inputs.start_vectors(1, ctx.npw(), 1)
    y = ctx.orthonormalize(torch.from_numpy(x).cuda()).cpu().numpy()
    low = np.linalg.cholesky(np.conj(x) @ x.T)
    ref = np.linalg.solve(np.conj(low), x)
    # both factorisations err by n eps kappa(S) at most, kappa about 1 + 0.3^2 n here
    tol = 4 * n * 2.0 ** -52 * (1 + 0.09 * n)
    assert np.linalg.norm(y - ref) <= tol * np.linalg.norm(ref)
    bad = x.copy()
    bad[n - 2] = 0  # its pivot is zero exactly, in whichever block it falls
    with pytest.raises(paro.ParoError):
        ctx.orthonormalize(torch.from_numpy(bad).cuda())
