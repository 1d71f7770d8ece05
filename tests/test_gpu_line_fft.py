"""Every cubic grid with a line-FFT form (csrc/fft_tile.cuh, hpsi_passes_reg.cuh): H psi and the density in FP64
and FP32 against the oracle, with rows and potentials of very different size."""
import numpy as np
import pytest
import torch

from oracle import pw
from paper_1702_04045_gb300 import inputs, paro

pytestmark = pytest.mark.gpu

L = 6.0
ECUT = {27: 20.2, 32: 27.2, 36: 35.4, 48: 48.0, 54: 80.6, 64: 108.4, 72: 141.4, 81: 179.0, 96: 234.0, 108: 330.0}


def _setup(n, precision):
    lat = np.eye(3) * L
    pos = np.array([[0.3, 0.2, 0.1], [3.1, 2.7, 3.3]])
    ecut = ECUT[n]
    ctx = paro.Context(lat, pos, ecut, 3, 2, precision)
    ctx.set_local_pp(**inputs.LOCAL_PP)
    assert ctx.grid == (n, n, n)
    b = pw.Basis(lat, ecut, ctx.grid)
    return ctx, b, pw.vloc_real(lat, pos, ctx.grid, ecut, **inputs.LOCAL_PP)


@pytest.mark.parametrize("n", sorted(ECUT))
def test_hpsi_on_every_grid(n):
    ctx, b, v = _setup(n, "fp64")
    psi = inputs.start_vectors(3, b.npw, n) / (1.0 + b.kin) * np.array([[1.0], [1e-9], [1e7]])
    ref = pw.apply_h(b, v, psi)
    got = ctx.apply_h(torch.from_numpy(psi).cuda()).cpu().numpy()
    # lines rounded to 2^-53 of their norm in six passes of at most eight roundings, against NumPy's own FFT error
    norm = np.linalg.norm(b.kin * psi, axis=1) + np.abs(v).max() * np.linalg.norm(psi, axis=1)
    assert (np.linalg.norm(got - ref, axis=1) <= 48 * 2.0 ** -53 * norm).all()
    got32 = ctx.apply_h(torch.from_numpy(psi.astype(np.complex64)).cuda()).cpu().numpy()
    assert (np.linalg.norm(got32 - ref, axis=1) <= 48 * 2.0 ** -24 * norm).all()


@pytest.mark.parametrize("n", sorted(ECUT))
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_density_on_every_grid(n, precision):
    ctx, b, _ = _setup(n, precision)
    ctx.set_orbitals(inputs.start_vectors(3, b.npw, n) / (1.0 + b.kin))
    rho = ctx.density().cpu().numpy()
    ref = 2.0 * (np.abs(pw.to_real_space(b, ctx.get_orbitals()[:2])) ** 2).sum(axis=0) / b.omega
    eps = 2.0 ** -53 if precision == "fp64" else 2.0 ** -24
    assert np.linalg.norm(rho - ref) <= 64 * eps * np.linalg.norm(ref)


@pytest.mark.parametrize("n", [27, 72])
def test_zero_and_nonfinite_rows(n):
    ctx, b, _ = _setup(n, "fp64")
    psi = torch.from_numpy(inputs.start_vectors(3, b.npw, n)).cuda()
    psi[0] = 0
    psi[1, 7] = complex(float("inf"), 0.0)
    out = ctx.apply_h(psi)
    assert (out[0] == 0).all()
    assert torch.isnan(torch.view_as_real(out[1])).any()
    assert torch.isfinite(torch.view_as_real(out[2])).all()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_batch_on_the_callers_arrays(precision):
    """paro_batch_apply_h reads and writes the caller's arrays where they allow it (their own outputs included) and
    goes through its own buffers where outputs overlap other inputs: the same values either way."""
    import ctypes
    ctxs, rows = [], []
    dt = torch.complex128 if precision == "fp64" else torch.complex64
    for i, ecut in enumerate((20.2, 48.0, 20.2)):
        ctx = paro.Context(np.eye(3) * L, np.array([[0.3 + 0.1 * i, 0.2, 0.1]]), ecut, 3, 2, precision)
        ctx.set_local_pp(**inputs.LOCAL_PP)
        ctxs.append(ctx)
        rows.append(torch.from_numpy(inputs.start_vectors(3, ctx.npw(), 40 + i)).to(dt).cuda())
    b = paro.Batch(ctxs)
    want = [c.apply_h(x) for c, x in zip(ctxs, rows)]
    tol = 1e-14 if precision == "fp64" else 1e-6

    def call(src, dst):
        p = (ctypes.c_void_p * 3)(*[t.data_ptr() for t in src])
        q = (ctypes.c_void_p * 3)(*[t.data_ptr() for t in dst])
        assert b.lib.paro_batch_apply_h(b.h, 0 if precision == "fp64" else 1, p, q) == 0
        for w, t in zip(want, dst):
            assert (torch.linalg.vector_norm(t - w) / torch.linalg.vector_norm(w)).item() < tol

    call(rows, [torch.empty_like(x) for x in rows])
    own = [x.clone() for x in rows]
    call(own, own)  # in place
    swapped = [x.clone() for x in rows]
    call(swapped, [swapped[2], torch.empty_like(rows[1]), swapped[0]])  # outputs over other problems' inputs


@pytest.mark.parametrize("n", [32, 36, 48, 72])
def test_state_of_the_fp64_iteration(n):
    """H psi as the FP64 iteration forms it (csrc/fft_reg.cuh, FP64 lines): the Ritz values and the vanishing
    off-diagonal elements of H over the orbitals against the oracle's H."""
    ctx, b, v = _setup(n, "fp64")
    ctx.set_orbitals(inputs.start_vectors(3, b.npw, n) / (1.0 + b.kin))
    psi = ctx.get_orbitals()
    h = psi.conj() @ pw.apply_h(b, v, psi).T
    norm = np.linalg.norm(b.kin * psi, axis=1).max() + np.abs(v).max()
    # the bound of an H psi above, twice: H of the orthonormal rows, and the rows' own rounding and rotation
    assert np.abs(h - np.diag(ctx.eigenvalues()[0])).max() <= 96 * 2.0 ** -53 * norm
