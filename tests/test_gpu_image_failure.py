"""A failure while the projectors' images (digit images, and the TF32 images of the inner solves) are formed leaves no half-formed images behind: the call that met it
reports it, and the next one, which finds nothing in its way, returns the right values. The failure is an error that
another part of the process left pending in the CUDA runtime (an allocation refused), which the library's first check
after a launch picks up."""
import ctypes
import re

import pytest

from paper_1702_04045_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision,dtype,tol,form", [("fp64", torch.complex128, 1e-12, 0),
                                                      ("mixed", torch.complex64, 2e-6, 0),
                                                      ("mixed", torch.complex64, 3e-5, 1)])
def test_products_after_a_failure_are_right(precision, dtype, tol, form):
    from paper_1702_04045_gb300 import paro

    def context():
        ctx = paro.context_from_config("si64_scf", precision)
        return ctx, torch.from_numpy(inputs.start_vectors(144, ctx.npw(), 3)).to(dtype).cuda()

    ctx, x = context()
    ref = ctx.apply_vnl(x, form).clone()
    ctx.close()
    ctx, x = context()
    out = torch.empty_like(x)
    torch.cuda.synchronize()
    lib = re.search(r"\S*libcudart\.so\S*", open("/proc/self/maps").read())
    if not lib:
        pytest.skip("the CUDA runtime is linked statically")
    rt = ctypes.CDLL(lib.group(0))
    ptr = ctypes.c_void_p()

    def call():
        return ctx.lib.paro_apply_vnl(ctx.h, 0, x.shape[0], paro.PARO_C64 if tol == 1e-12 else paro.PARO_C32,
                                      ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(out.data_ptr()), form)

    assert rt.cudaMalloc(ctypes.byref(ptr), ctypes.c_size_t(1 << 60)) != 0
    first = call()
    rt.cudaGetLastError()  # for torch, should the library not have met it
    assert first in (paro.PARO_OK, paro.PARO_ERR_CUDA)
    for _ in range(2):
        assert call() == paro.PARO_OK
        assert float((out - ref).abs().max()) < tol * float(ref.abs().max())
