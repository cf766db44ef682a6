"""Memory that outlives a handle: it goes back to the driver when asked for and before an allocation fails, and scratch
memory is clear when the call that reserves it returns."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _kept_memory(nm):
    """Leaves some 100 MB of a freed handle with the library; returns the free bytes of the device with them out."""
    nm.nm_memory_trim()
    w = torch.randn((1024, 3, 3, 1024), device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    nm.nm_prune(w, 1, 4, 64).free()
    assert torch.cuda.mem_get_info()[0] <= free - (64 << 20)
    return free


def test_trim_returns_the_memory_of_freed_handles():
    from paper_2507_17301_b200 import nm
    free = _kept_memory(nm)
    nm.nm_memory_trim()
    assert torch.cuda.mem_get_info()[0] >= free


def test_kept_memory_goes_back_before_a_reservation_fails():
    from paper_2507_17301_b200 import nm
    small = nm.nm_prune(torch.randn((16, 1, 1, 16), device="cuda"), 2, 4, 16)
    free = _kept_memory(nm)
    with pytest.raises(nm.NmError) as e:
        nm.nm_weights_reserve(small, 1 << 50)
    assert e.value.status == nm.NM_ERR_ALLOC
    assert torch.cuda.mem_get_info()[0] >= free


def test_reserved_scratch_is_cleared_when_the_call_returns():
    """A launch on a stream that does not wait for the default one may follow at once."""
    from paper_2507_17301_b200 import nm
    hnd = nm.nm_prune(torch.randn((16, 1, 1, 16), device="cuda"), 2, 4, 16)
    torch.cuda.synchronize()
    nm.nm_weights_reserve(hnd, 4 << 30)
    assert torch.cuda.default_stream().query()
    hnd.free()
