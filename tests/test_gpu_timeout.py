"""Bounded waits of the sliced products that give up are reported: with PARO_SLICE_POLLS=0 every such wait gives up
at once (the kernel drains what it started and returns), the calls that wait for the GPU return PARO_ERR_TIMEOUT,
and an enqueue-only call is reported by the next one that waits, once."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")

CODE = r"""
import numpy as np, torch
from paper_1702_04045_gb300 import inputs, paro

lat, pos = inputs.diamond_cell(1, 10.26, 91)

def context(precision="fp64"):
    ctx = paro.Context(lat, pos, 5.0, 4, 4, precision)
    ctx.set_local_pp(**inputs.LOCAL_PP)
    ctx.set_kb(inputs.KB_RC, inputs.kb_strengths(len(pos), 92))
    return ctx

def status(f):
    try:
        f()
    except paro.ParoError as e:
        return e.status
    return paro.PARO_OK

ctx = context()
x = torch.from_numpy(inputs.start_vectors(4, ctx.npw(), 7)).cuda()
y = torch.empty_like(x)
print(status(lambda: ctx.orthonormalize(x)),
      status(lambda: ctx.solve_source(np.zeros(4), x, 0.1, 3)),
      status(lambda: ctx.apply_vnl(x)),
      status(lambda: ctx.apply_h(x)),                                     # enqueued only
      status(lambda: ctx.orthonormalize(x.to(torch.complex64))),          # reports it
      status(lambda: ctx.orthonormalize(x.to(torch.complex64))),          # once
      status(lambda: ctx.apply_h_adjoint(x, y.copy_(x), grads=("pos",))),  # enqueued only
      status(lambda: ctx.orthonormalize(x.to(torch.complex64))))
# the FP64 iteration has no such wait; its energy does
ctx = context()
ctx.set_orbitals(inputs.start_vectors(4, ctx.npw(), 7))
print(status(lambda: ctx.step(1, 0.25, 2)), status(ctx.energy), status(lambda: ctx.step(1, 0.25, 2)))
"""


def test_timeouts_are_reported():
    ok, to = 0, -5  # PARO_OK, PARO_ERR_TIMEOUT
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, PARO_SLICE_POLLS="0"))
    assert r.returncode == 0, r.stderr
    got = [[int(v) for v in line.split()] for line in r.stdout.strip().splitlines()]
    assert got == [[to, to, to, ok, to, ok, ok, to], [ok, to, ok]]
    # and none of it happens with the usual limit
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=300,
                       env={k: v for k, v in os.environ.items() if k != "PARO_SLICE_POLLS"})
    assert r.returncode == 0, r.stderr
    assert {int(v) for v in r.stdout.split()} == {ok}
