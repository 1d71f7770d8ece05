"""Four-digit form of the FP32 nonlocal term (csrc/k_slice.cu) on the 64-atom cell against FP64 products of the
same FP32 operands: both column tiles (48 and 64), whole and partial, rows of very different size, and non-finite
rows."""
import numpy as np
import pytest

from oracle import pw
from paper_1702_04045_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def si64():
    from paper_1702_04045_gb300 import paro
    ctx = paro.context_from_config("si64_scf", "mixed")
    lat, pos, d, c = inputs.config_inputs("si64_scf")
    b = pw.Basis(lat, c["ecut"], ctx.grid)
    beta = pw.kb_beta(lat, pos, b.q, inputs.KB_RC).astype(np.complex64).astype(np.complex128)
    return ctx, torch.from_numpy(beta).cuda(), torch.from_numpy(pw.kb_dvec(d)).cuda()


# 48-column tiles take 32, 48, 65 and 133 rows, 64-column tiles 49, 64, 97 and 192
@pytest.mark.parametrize("nb", [32, 48, 49, 64, 65, 97, 133, 192])
def test_vnl_f32_by_digits(si64, nb):
    ctx, beta, dvec = si64
    npj, npw = beta.shape
    assert npj * nb * npw >= 1.5e8  # the digit slices' side of their rule
    rng = np.random.default_rng(nb)
    scale = 10.0 ** rng.uniform(-14, 8, size=(nb, 1))
    psi = (inputs.start_vectors(nb, npw, nb) * scale).astype(np.complex64)
    bad = nb // 2
    psi[bad, 17] = np.inf if nb % 2 else np.nan
    x = torch.from_numpy(psi).cuda()
    got = ctx.apply_vnl(x)
    assert torch.isnan(torch.view_as_real(got[bad])).all()
    keep = torch.tensor([i for i in range(nb) if i != bad]).cuda()
    xd = x[keep].to(torch.complex128)
    proj = beta.conj() @ xd.T
    ref = (beta.T @ (dvec[:, None] * proj)).T
    # operands of both products to 2^-31 of their rows' largest value, the library's FP32 table against the oracle's
    # (2^-24), the result rounded to FP32 twice (2^-24): together below 2^-22 of sum_p |beta_p| |D_p| |P_p|, and the
    # operands' part below 2^-30 max|beta| |psi|_1 a projection
    ab = beta.abs()
    mag = (ab.T @ (dvec.abs()[:, None] * proj.abs())).T
    low = float(dvec.abs().max()) * ab.sum(0)[None, :] * ab.max() * xd.abs().sum(1)[:, None]
    assert ((got[keep].to(torch.complex128) - ref).abs() <= 2.0 ** -22 * mag + 2.0 ** -30 * low).all()
