"""The sliced products' kernel when its bounded waits give up (PARO_SLICE_POLLS: polls until then): it drains the
copies and MMAs it started, releases tensor memory and reports, so that the call returns PARO_ERR_TIMEOUT and the
context, whose next products run on the CUDA cores, stays usable. With a few polls a wait may or may not give up:
the call then reports it or is right."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")

CODE = r"""
import numpy as np, torch
from oracle import pw
from paper_1702_04045_gb300 import inputs, paro

lat, pos = inputs.diamond_cell(1, 10.26, 91)
d = inputs.kb_strengths(len(pos), 92)

def one(n):
    ctx = paro.Context(lat, pos, 5.0, 4, 4, "fp64")
    ctx.set_local_pp(**inputs.LOCAL_PP)
    ctx.set_kb(inputs.KB_RC, d)
    b = pw.Basis(lat, 5.0, ctx.grid)
    beta = pw.kb_beta(lat, pos, b.q, inputs.KB_RC)
    psi = inputs.start_vectors(n, b.npw, n)
    ref = (beta.T @ (pw.kb_dvec(d)[:, None] * (np.conj(beta) @ psi.T))).T
    x = torch.from_numpy(psi).cuda()
    try:
        out = ctx.apply_vnl(x)
        ok = np.abs(out.cpu().numpy() - ref).max() < 1e-12 * np.abs(ref).max()
        status = paro.PARO_OK if ok else "wrong"
    except paro.ParoError as e:
        status = e.status
    small = ctx.apply_h(x.to(torch.complex64)).cpu().numpy()
    h = pw.apply_h(b, pw.vloc_real(lat, pos, ctx.grid, 5.0, **inputs.LOCAL_PP), psi, beta, pw.kb_dvec(d))
    assert np.abs(small - h).max() < 2e-6 * np.abs(h).max()
    return status

print(one(1), one(33), one(160))
"""


@pytest.mark.parametrize("polls,allowed", [("0", {"-5"}), ("1", {"-5", "0"}), ("8", {"-5", "0"}), (None, {"0"})])
def test_a_given_up_wait_is_drained_and_reported(polls, allowed):
    env = {k: v for k, v in os.environ.items() if k != "PARO_SLICE_POLLS"}
    if polls is not None:
        env["PARO_SLICE_POLLS"] = polls
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=300, env=env)
    assert r.returncode == 0, r.stderr
    assert set(r.stdout.split()) <= allowed, r.stdout
