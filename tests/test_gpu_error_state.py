"""A call that fails for want of device memory reports it and leaves no error behind: torch, another context, and the
same context go on once memory is free."""
import pytest

from paper_1702_04045_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_a_refused_allocation_is_reported_once():
    from paper_1702_04045_gb300 import paro

    ctx = paro.context_from_config("si64_scf", "fp64")
    x = torch.from_numpy(inputs.start_vectors(144, ctx.npw(), 3)).cuda()
    ref = ctx.orthonormalize(x)
    ones = torch.ones(8, device="cuda")
    assert float((ones + ones).sum()) == 16.0  # torch's kernels are loaded while there is memory for them
    ctx.close()
    ctx = paro.context_from_config("si64_scf", "fp64")
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - (32 << 20), dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(paro.ParoError) as e:
            ctx.orthonormalize(x, out=y)  # a copy of the rows alone is 55 MB
        assert e.value.status == paro.PARO_ERR_CUDA and "out of memory" in str(e.value)
        assert float((ones + ones).sum()) == 16.0
    finally:
        del filler
        torch.cuda.empty_cache()
    other = paro.context_from_config("si64_scf", "mixed")
    other.apply_h(x.to(torch.complex64))
    assert torch.equal(ctx.orthonormalize(x, out=y), ref)
