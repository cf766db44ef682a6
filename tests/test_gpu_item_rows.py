"""The expanded-operand kernel's work items of fewer than 128 pixels (chosen where the items do not fill whole rounds of
the SMs): several rounds, boxes of fewer than 32 pixels at an item's end, a ragged last item, the fused shortcut, two
channel slices; bit for bit on integer inputs."""
import numpy as np
import pytest
import torch

import oracle
from paper_2507_17301_b200 import inputs
from paper_2507_17301_b200.inputs import ConvShape

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s", [
    ConvShape("rounds_1x1", 8, 56, 56, 32, 32, 1, 1, 1, 0, 1, 2, 4, 16),        # 196 items of 128 on 148 SMs: two rounds
    ConvShape("slices_1x1", 8, 56, 56, 32, 64, 1, 1, 1, 0, 1, 2, 4, 32),        # two slices of 32: three rounds
    ConvShape("ragged_3x3", 9, 47, 45, 32, 32, 3, 3, 1, 1, 1, 2, 4, 16),        # 19035 pixels
    ConvShape("strided_3x3", 5, 93, 91, 32, 64, 3, 3, 2, 1, 1, 1, 4, 64),
    ConvShape("one_round", 1, 41, 40, 64, 32, 1, 1, 1, 0, 1, 2, 4, 16),         # fewer items than SMs: 32-pixel items
    ConvShape("padded_channels", 3, 61, 60, 36, 28, 1, 1, 1, 0, 1, 2, 4, 4),
], ids=lambda s: s.name)
@pytest.mark.parametrize("residual", [False, True])
def test_items_of_any_size(s, residual):
    from paper_2507_17301_b200 import nm
    w, x, b = inputs.make_int_case(s)
    vr, ir = oracle.prune(w.numpy(), s.n_keep, s.m_group, s.tile_t)
    geom = ((s.stride,) * 2, (s.pad,) * 2, (s.dil,) * 2)
    res = torch.randint(-9, 10, (s.batch, s.ho, s.wo, s.c_out), generator=torch.Generator().manual_seed(1)).float() if residual else None
    if residual:
        yr = oracle.conv2d_res(vr, ir, s.kh, s.kw, s.c_in, s.tile_t, x.numpy(), *geom, b.numpy(), res.numpy(), True)
    else:
        yr = oracle.conv2d(vr, ir, s.kh, s.kw, s.c_in, s.tile_t, x.numpy(), *geom, b.numpy(), True)
    hnd = nm.nm_prune(w.cuda(), s.n_keep, s.m_group, s.tile_t)
    ran = 0
    for bn in (32, 64):
        for split in (0, 1):
            for kblk in (1, 2):
                plan = nm.nm_plan_t()
                plan.variant, plan.bn, plan.split, plan.kblk = 4, bn, split, kblk
                try:
                    y = nm.nm_conv2d(hnd, x.cuda(), s.kh, s.kw, s.stride, s.pad, s.dil, b.cuda(), True, plan=plan,
                                     residual=res.cuda() if residual else None)
                except nm.NmError as e:
                    if e.status == nm.NM_ERR_UNSUPPORTED:
                        continue
                    raise
                nm.nm_weights_check(hnd)
                assert np.array_equal(y.cpu().numpy(), yr), plan.as_dict()
                ran += 1
    assert ran >= 2


@pytest.mark.parametrize("c_out,bn", [(96, 96), (160, 160), (320, 160), (32, 32)])
def test_odd_numbers_of_channel_blocks(c_out, bn):
    """Warps that take every other block change places from item to item: several items per CTA, with and without a shortcut."""
    from paper_2507_17301_b200 import nm
    s = ConvShape("odd_blocks", 9, 57, 59, 32, c_out, 1, 1, 1, 0, 1, 2, 4, 32)      # 237 blocks of 128 pixels
    w, x, b = inputs.make_int_case(s)
    vr, ir = oracle.prune(w.numpy(), s.n_keep, s.m_group, s.tile_t)
    geom = ((1, 1), (0, 0), (1, 1))
    res = torch.randint(-9, 10, (s.batch, s.h, s.w, c_out), generator=torch.Generator().manual_seed(1)).float()
    hnd = nm.nm_prune(w.cuda(), s.n_keep, s.m_group, s.tile_t)
    yr = oracle.conv2d(vr, ir, 1, 1, s.c_in, s.tile_t, x.numpy(), *geom, b.numpy(), True)
    yres = oracle.conv2d_res(vr, ir, 1, 1, s.c_in, s.tile_t, x.numpy(), *geom, b.numpy(), res.numpy(), True)
    for split in (0, 1):
        plan = nm.nm_plan_t()
        plan.variant, plan.bn, plan.split = 4, bn, split
        for r, want in ((None, yr), (res.cuda(), yres)):
            y = nm.nm_conv2d(hnd, x.cuda(), 1, 1, 1, 0, 1, b.cuda(), True, plan=plan, residual=r)
            nm.nm_weights_check(hnd)
            assert np.array_equal(y.cpu().numpy(), want), (split, r is not None)
