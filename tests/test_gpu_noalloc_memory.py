"""paro_apply_h_noalloc leaves device memory alone: free memory is the same before and after the first call on a
context and a larger second one, with projectors, in both data types. On the 64-atom cell any workspace that the
projector products would take is far above the allocator's granularity (2 MiB)."""
import pytest

from paper_1702_04045_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dtype", [torch.complex128, torch.complex64])
def test_noalloc_keeps_free_memory(precision, dtype):
    from paper_1702_04045_gb300 import paro

    def context():
        ctx = paro.context_from_config("si64_scf", precision)
        return ctx, torch.from_numpy(inputs.start_vectors(8, ctx.npw(), 4)).to(dtype).cuda()

    # another context loads the kernels first: loading a kernel takes device memory of its own
    ctx, psi = context()
    ctx.apply_h_noalloc(psi, torch.empty_like(psi))
    ctx.close()
    ctx, psi = context()
    out = torch.empty_like(psi)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for nb in (2, 8):
        ctx.apply_h_noalloc(psi[:nb], out[:nb])
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] == free
    ref = ctx.apply_h(psi)
    assert float((out - ref).abs().max() / ref.abs().max()) < (1e-12 if dtype == torch.complex128 else 2e-6)
