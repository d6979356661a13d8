"""What the library's memory pool keeps: a destroyed target's memory is back with the
device when the call returns, but for the 256 MB the pool may keep for its next calls."""
import pytest

pytestmark = pytest.mark.gpu

KEEP = 256 << 20
CHUNK = 32 << 20   # the driver hands memory to a pool in pieces of this size


@pytest.fixture(scope="module")
def fr():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2007_07627_gb300 import build
    build.build()
    import paper_2007_07627_gb300 as fr
    fr.lib()
    return fr


def test_a_destroyed_targets_memory_is_free_again(fr):
    import torch
    n = 40_000_000                                # its index takes over 1 GB
    q = torch.rand((n, 3), device="cuda")
    fr.target_create(q[:1000].contiguous()).destroy()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    t = fr.target_create(q)
    held = before - torch.cuda.mem_get_info()[0]
    t.destroy()
    after = torch.cuda.mem_get_info()[0]
    assert held > 2 * (KEEP + CHUNK)
    assert before - after <= KEEP + CHUNK
