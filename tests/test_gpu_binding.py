"""What the native argument marshalling passes on: torch's own exception types."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_2505_01068_b200 as lib
    lib.load()
    return lib


def test_failed_allocation_raises_torch_out_of_memory_error(g):
    """Callers catch torch.OutOfMemoryError to go on with a smaller batch.  The limit is one of this process's allocator."""
    seg, d = (1024, 2048, 1024), 512
    x = torch.zeros((8, sum(seg), d), device="cuda", dtype=torch.bfloat16)
    w = torch.zeros((3 * d, d), device="cuda", dtype=torch.bfloat16)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + (16 << 20)) / torch.cuda.get_device_properties(0).total_memory)
    try:
        with pytest.raises(torch.OutOfMemoryError):
            g.im_qkv_proj(x, w, None, seg, 8)                       # the result is 100 MB
        half = g.im_qkv_proj(x[:1, :], w, None, seg, 8)             # 12.6 MB: fits
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert bool((half == 0).all()) and g.last_device_status() == (0, 0)
