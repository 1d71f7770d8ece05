"""Products that keep digit images of their operands do without them when device memory is short: the calls take the
plain products and return the same values. Each call runs once with memory free, which says what it takes; a fresh
context then finds `spare` bytes less than that."""
import numpy as np
import pytest

from paper_1702_04045_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MIB = 1 << 20


def _vnl(ctx, x):
    return ctx.apply_vnl(x)


def _orth(ctx, x):
    return ctx.orthonormalize(x)


def _adjoint(ctx, x):
    return ctx.apply_h_adjoint(x, torch.flip(x, (0,)), grads=("pos",))[2]


# spare: well below what the images (vnl: at least 32 bytes an entry of 256 x 23847; orth: 70 bytes an entry of
# 144 x 23847) and the adjoint's six weighted blocks (five of them 137 MB) take
@pytest.mark.parametrize("call,precision,dtype,spare,tol", [
    (_vnl, "fp64", torch.complex128, 200 * MIB, 1e-12), (_vnl, "mixed", torch.complex64, 100 * MIB, 2e-6),
    (_orth, "fp64", torch.complex128, 100 * MIB, 1e-12), (_adjoint, "mixed", torch.complex64, 64 * MIB, 2e-5)])
def test_calls_do_without_optional_memory(call, precision, dtype, spare, tol):
    from paper_1702_04045_gb300 import paro

    def context():
        ctx = paro.context_from_config("si64_scf", precision)
        return ctx, torch.from_numpy(inputs.start_vectors(144, ctx.npw(), 3)).to(dtype).cuda()

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    ctx, x = context()
    call(ctx, x)  # loads the kernels and fills torch's pool
    ctx.close()
    ctx, x = context()
    before = free()
    ref = call(ctx, x).cpu()
    taken = before - free()
    ctx.close()
    assert taken > spare
    ctx, x = context()
    filler = torch.empty(free() - taken + spare, dtype=torch.uint8, device="cuda")
    try:
        got = call(ctx, x).cpu()
        again = call(ctx, x).cpu()
    finally:
        del filler
        torch.cuda.empty_cache()
    assert float((got - ref).abs().max()) < tol * float(ref.abs().max())
    assert torch.equal(got, again)
    # with the memory back, the same context takes the usual products again
    assert torch.equal(call(ctx, x).cpu(), ref)


def test_own_allocations_take_the_images_back():
    """A context that holds images (342 MB for the projectors alone) and finds 48 MB free still takes orbitals, whose
    two arrays are 110 MB, with the workspaces of their Rayleigh-Ritz step."""
    from paper_1702_04045_gb300 import paro

    def context():
        ctx = paro.context_from_config("si64_scf", "fp64")
        return ctx, inputs.start_vectors(144, ctx.npw(), 3)

    ctx, x = context()
    ctx.set_orbitals(x)
    ref = ctx.eigenvalues()
    ctx.close()
    ctx, x = context()
    ctx.apply_vnl(torch.from_numpy(x).cuda())
    torch.cuda.synchronize()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - 48 * MIB, dtype=torch.uint8, device="cuda")
    try:
        ctx.set_orbitals(x)
    finally:
        del filler
        torch.cuda.empty_cache()
    assert np.array_equal(ctx.eigenvalues(), ref)
