"""The cluster kernel (plan.variant = 10) against the CPU oracle, bit for bit on integer inputs: the three forms of its
activation loads, one to eight ranges of the reduction axis, every tile width, ragged items, a ring shorter than a range,
channel counts that end inside a block, the fused shortcut."""
import numpy as np
import pytest
import torch

import oracle
from paper_2507_17301_b200.inputs import ConvShape
from parity import assert_conv_close, gpu_layer, oracle_layer, tensors_for

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nm():
    from paper_2507_17301_b200 import nm as mod
    return mod


def _plans(nm, stages=(0,)):
    for bn in (32, 64, 128):
        for cs in (1, 2, 4, 8):
            for st in stages:
                p = nm.nm_plan_t()
                p.variant, p.bn, p.ksplit, p.stages = 10, bn, cs, st
                yield p


SHAPES = [
    ConvShape("box_7x7", 1, 7, 7, 128, 128, 3, 3, 1, 1, 1, 2, 4, 32),          # small input: boxes of output rows
    ConvShape("box_rows", 2, 13, 11, 32, 64, 3, 3, 1, 1, 1, 1, 4, 16),         # 11 rows an item fit, 13 are needed: 7 + 6
    ConvShape("box_dil_nopad", 1, 15, 17, 64, 32, 3, 3, 1, 0, 2, 2, 4, 16),
    ConvShape("rows_1x1", 1, 7, 7, 512, 96, 1, 1, 1, 0, 1, 2, 8, 8),           # 49 pixels: 56-row boxes
    ConvShape("rows_1x1_odd", 3, 9, 9, 144, 60, 1, 1, 1, 0, 1, 3, 4, 5),       # blocks ending inside 32 channels, both sides
    ConvShape("im2col_14", 1, 14, 14, 256, 64, 3, 3, 1, 1, 1, 2, 4, 64),       # 196 pixels = 2 items of 104 rows
    ConvShape("im2col_s2", 3, 28, 28, 64, 128, 3, 3, 2, 1, 1, 2, 4, 64),
    ConvShape("im2col_1x1_s2", 1, 29, 31, 68, 32, 1, 1, 2, 0, 1, 2, 4, 16),
    ConvShape("im2col_5x5", 1, 24, 24, 64, 32, 5, 5, 1, 2, 1, 2, 8, 16),
]


@pytest.mark.parametrize("s", SHAPES, ids=lambda s: s.name)
def test_cluster_kernel_integer_exact(nm, s):
    w, x, b = tensors_for(s, True)
    _, _, yr = oracle_layer(s, w, x, b)
    ran = 0
    for plan in _plans(nm, (0, 2)):
        try:
            _, _, _, y = gpu_layer(nm, s, w, x, b, True, plan)
        except nm.NmError as e:
            if e.status == nm.NM_ERR_UNSUPPORTED:
                continue
            raise
        ran += 1
        assert np.array_equal(y, yr), plan.as_dict()
    assert ran >= 4   # one width, one or two ranges, two rings at least


@pytest.mark.parametrize("s", SHAPES[:1] + SHAPES[4:6], ids=lambda s: s.name)
def test_cluster_kernel_shortcut_and_repeat(nm, s):
    """act(conv + bias + shortcut), launched back to back on one stream (the next launch's CTAs start early): every output
    equals the first, bit for bit, and the oracle's within the tolerance of TF32."""
    w, x, b = tensors_for(s)
    res = torch.randn((s.batch, s.ho, s.wo, s.c_out), generator=torch.Generator().manual_seed(3))
    vr, ir = oracle.prune(w.numpy(), s.n_keep, s.m_group, s.tile_t)
    yr = oracle.conv2d_res(vr, ir, s.kh, s.kw, s.c_in, s.tile_t, x.numpy(), (s.stride,) * 2, (s.pad,) * 2, (s.dil,) * 2, b.numpy(),
                           res.numpy(), True)
    hnd = nm.nm_prune(w.cuda(), s.n_keep, s.m_group, s.tile_t)
    xd, bd, rd = x.cuda(), b.cuda(), res.cuda()
    for plan in _plans(nm):
        try:
            ys = [nm.nm_conv2d(hnd, xd, s.kh, s.kw, s.stride, s.pad, s.dil, bd, True, plan=plan, residual=rd) for _ in range(6)]
        except nm.NmError as e:
            if e.status == nm.NM_ERR_UNSUPPORTED:
                continue
            raise
        nm.nm_weights_check(hnd)
        assert_conv_close(ys[0].cpu().numpy(), yr)
        assert all(torch.equal(y, ys[0]) for y in ys[1:]), plan.as_dict()


def test_plans_it_does_not_take(nm):
    s = SHAPES[0]
    w, x, b = tensors_for(s, True)
    for field, value in (("ksplit", 3), ("ksplit", 16), ("bn", 48), ("stages", 1), ("stages", 13)):
        plan = nm.nm_plan_t()
        plan.variant, plan.bn, plan.ksplit = 10, 32, 2
        setattr(plan, field, value)
        with pytest.raises(nm.NmError) as e:
            gpu_layer(nm, s, w, x, b, True, plan)
        assert e.value.status == nm.NM_ERR_UNSUPPORTED
