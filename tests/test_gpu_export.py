"""Export of a handle's canonical arrays: one launch where both destinations are 16-byte aligned, copies where they are not, sizes that
are no multiple of 16 bytes; and layouts that are written in full without being cleared first, on memory of earlier handles."""
import ctypes

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,n,m,t", [((3, 1, 1, 5), 1, 2, 2), ((33, 3, 3, 7), 2, 5, 8), ((64, 3, 3, 64), 2, 4, 64), ((128, 1, 1, 96), 3, 4, 32)])
@pytest.mark.parametrize("shift", [0, 1])
def test_export_matches_the_oracle(shape, n, m, t, shift):
    from paper_2507_17301_b200 import nm
    torch.manual_seed(3)
    w = torch.randn(shape)
    vr, ir = oracle.prune(w.numpy(), n, m, t)
    hnd = nm.nm_prune(w.cuda(), n, m, t)
    v, i = nm.nm_weights_export(hnd)
    assert np.array_equal(v.cpu().numpy(), vr) and np.array_equal(i.cpu().numpy(), ir)
    vb = torch.empty(vr.size + shift, device="cuda")
    ib = torch.empty(ir.size + 2 * shift, dtype=torch.uint16, device="cuda")
    nm._check(nm._lib.nm_weights_export(hnd.handle, ctypes.c_void_p(vb.data_ptr() + 4 * shift), ctypes.c_void_p(ib.data_ptr() + 4 * shift), nm._stream()))
    torch.cuda.synchronize()
    assert np.array_equal(vb.cpu().numpy()[shift:].reshape(vr.shape), vr) and np.array_equal(ib.cpu().numpy()[2 * shift:].reshape(ir.shape), ir)


@pytest.mark.parametrize("n,m", [(2, 4), (1, 4), (2, 8), (1, 8), (3, 4)])
def test_layouts_on_used_memory(n, m):
    """A handle's block may come from an earlier handle: what is not cleared must be written."""
    from paper_2507_17301_b200 import nm
    g = torch.Generator().manual_seed(5)
    x = torch.randint(-3, 4, (2, 16, 16, 64), generator=g).float()
    for _ in range(2):
        used = nm.nm_prune(torch.full((64, 3, 3, 64), float("inf"), device="cuda"), n, m, 32)
        used.free()
        w = torch.randint(-3, 4, (64, 3, 3, 64), generator=g).float()
        vr, ir = oracle.prune(w.numpy(), n, m, 32)
        yr = oracle.conv2d(vr, ir, 3, 3, 64, 32, x.numpy(), (1, 1), (1, 1), (1, 1), None, False)
        hnd = nm.nm_prune(w.cuda(), n, m, 32)
        for variant in (1, 2, 3, 4, 8):
            plan = nm.nm_plan_t()
            plan.variant = variant
            y = nm.nm_conv2d(hnd, x.cuda(), 3, 3, 1, 1, 1, None, False, plan=plan)
            nm.nm_weights_check(hnd)
            assert np.array_equal(y.cpu().numpy(), yr), variant


@pytest.mark.parametrize("t", [1, 3, 8, 24])
def test_gather_layout_of_narrow_tiles_on_used_memory(t):
    """Rows of a tile only, a ragged last tile, retained columns that end inside a chunk; on memory of an earlier handle."""
    from paper_2507_17301_b200 import nm
    g = torch.Generator().manual_seed(6)
    x = torch.randint(-3, 4, (2, 9, 11, 20), generator=g).float()
    w = torch.randint(-3, 4, (50, 3, 3, 20), generator=g).float()
    vr, ir = oracle.prune(w.numpy(), 2, 4, t)
    yr = oracle.conv2d(vr, ir, 3, 3, 20, t, x.numpy(), (1, 1), (1, 1), (1, 1), None, False)
    plan = nm.nm_plan_t()
    plan.variant = 1
    for _ in range(2):
        nm.nm_prune(torch.full((50, 3, 3, 20), float("inf"), device="cuda"), 2, 4, t).free()
        hnd = nm.nm_prune(w.cuda(), 2, 4, t)
        y = nm.nm_conv2d(hnd, x.cuda(), 3, 3, 1, 1, 1, plan=plan)
        nm.nm_weights_check(hnd)
        assert np.array_equal(y.cpu().numpy(), yr)


def test_a_handle_of_one_channel_tiles_is_not_padded():
    """512 x 3 x 3 x 512 at 2:4, T = 1: values, gather and slab layouts 4.7 MB each, taps 4.7, expanded 9.4, indices 3.5: 32 MB."""
    from paper_2507_17301_b200 import nm
    w = torch.randn((512, 3, 3, 512), device="cuda")
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    hnd = nm.nm_prune(w, 2, 4, 1)
    assert before - torch.cuda.mem_get_info()[0] <= 36 << 20
    hnd.free()
