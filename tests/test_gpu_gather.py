"""The direct-gather kernel (plan.variant = 1) against the CPU oracle, bit for bit on integer inputs: tile widths below, at and
above a staging pass, odd ones, tails of tiles and channels, tap counts up to the mask's 64 and above (bounds by comparison), one to eight ranges of the
chunks, several passes per CTA, ragged pixel blocks that span images, the fused shortcut."""
import numpy as np
import pytest
import torch

import oracle
from paper_2507_17301_b200 import inputs
from paper_2507_17301_b200.inputs import ConvShape

pytestmark = pytest.mark.gpu

# name, batch, h, w, c_in, c_out, kh, kw, stride, pad, dil, N, M, T
SHAPES = [
    ConvShape("t1_odd", 2, 9, 7, 5, 7, 3, 3, 1, 1, 1, 2, 3, 1),
    ConvShape("t5_tail", 1, 20, 19, 13, 33, 3, 3, 2, 1, 1, 1, 4, 5),              # last tile of three channels
    ConvShape("t8", 3, 17, 15, 36, 40, 3, 3, 1, 1, 1, 2, 4, 8),
    ConvShape("t33", 1, 12, 12, 20, 70, 1, 1, 1, 0, 1, 3, 5, 33),
    ConvShape("t48_tail4", 2, 11, 11, 24, 52, 3, 3, 1, 2, 2, 2, 4, 48),           # a tile of four channels
    ConvShape("t100", 1, 10, 9, 16, 230, 3, 3, 1, 1, 1, 2, 4, 100),              # two passes per tile
    ConvShape("t256", 1, 8, 8, 12, 300, 1, 3, 1, 1, 1, 2, 4, 256),
    ConvShape("t128_cout52", 1, 8, 37, 20, 52, 3, 3, 1, 1, 1, 4, 8, 128),         # tile wider than the layer
    ConvShape("k7x7", 2, 15, 14, 6, 24, 7, 7, 2, 3, 1, 2, 4, 8),                  # 49 taps
    ConvShape("k5x7_dil", 1, 19, 23, 8, 16, 5, 7, 1, 2, 2, 2, 4, 16),             # 35 taps
    ConvShape("one_column", 1, 9, 9, 1, 4, 1, 1, 1, 0, 1, 1, 1, 4),
    ConvShape("images", 40, 3, 3, 18, 32, 3, 3, 1, 1, 1, 2, 4, 32),               # a block of 128 pixels spans 15 images
    ConvShape("split2", 1, 7, 7, 34, 32, 3, 3, 1, 1, 1, 2, 4, 32),                # five chunks
    ConvShape("split4", 1, 13, 13, 100, 60, 3, 3, 1, 1, 1, 2, 4, 12),
    ConvShape("split8", 1, 7, 7, 300, 50, 3, 3, 1, 1, 1, 2, 4, 50),
    ConvShape("split8_passes", 1, 6, 6, 300, 200, 3, 3, 1, 1, 1, 2, 4, 200),      # four passes through the exchange, ranks without rows
    ConvShape("split_ragged", 3, 34, 11, 75, 330, 3, 3, 1, 1, 1, 3, 4, 64),      # six tiles, the last block ragged
    ConvShape("split_7x7", 1, 9, 9, 30, 20, 7, 7, 1, 3, 1, 2, 4, 20),
    ConvShape("many_tiles", 6, 60, 60, 18, 72, 1, 1, 1, 0, 1, 2, 4, 4),           # 18 tiles
    ConvShape("wide_kept", 2, 30, 30, 10, 16, 3, 3, 1, 1, 1, 10, 10, 16),         # nothing pruned
    ConvShape("k8x8", 2, 13, 12, 6, 20, 8, 8, 1, 4, 1, 2, 4, 8),                  # 64 taps: the mask's last bit
    ConvShape("k9x9_s2", 2, 21, 19, 4, 24, 9, 9, 2, 4, 1, 2, 4, 8),               # 81 taps from here on: no mask
    ConvShape("k5x13_dil", 1, 24, 40, 7, 12, 5, 13, 1, 6, 2, 2, 7, 5),
    ConvShape("k1x65", 1, 3, 70, 3, 8, 1, 65, 1, 0, 1, 1, 3, 8),
    ConvShape("k9x9_images", 30, 5, 5, 6, 36, 9, 9, 1, 4, 1, 1, 4, 12),           # a block of 128 pixels spans six images, the last block ragged
    ConvShape("k9x9_split8", 1, 9, 9, 40, 72, 9, 9, 1, 4, 1, 2, 4, 72),           # 51 chunks over a cluster, two passes
    ConvShape("k11x11_split", 3, 14, 15, 16, 30, 11, 11, 2, 5, 1, 1, 8, 30),
]


@pytest.mark.parametrize("s", SHAPES, ids=lambda s: s.name)
@pytest.mark.parametrize("residual", [False, True])
def test_gather_kernel_integer_exact(s, residual):
    from paper_2507_17301_b200 import nm
    if residual and s.c_out % 4 != 0:
        pytest.skip("a shortcut input needs c_out % 4 == 0")
    w, x, b = inputs.make_int_case(s)
    vr, ir = oracle.prune(w.numpy(), s.n_keep, s.m_group, s.tile_t)
    geom = ((s.stride,) * 2, (s.pad,) * 2, (s.dil,) * 2)
    hnd = nm.nm_prune(w.cuda(), s.n_keep, s.m_group, s.tile_t)
    plan = nm.nm_plan_t()
    plan.variant = 1
    ho, wo = nm.out_shape(x.shape, s.kh, s.kw, s.c_out, *geom)[1:3]
    if residual:
        res = torch.randint(-9, 10, (s.batch, ho, wo, s.c_out), generator=torch.Generator().manual_seed(1)).float()
        yr = oracle.conv2d_res(vr, ir, s.kh, s.kw, s.c_in, s.tile_t, x.numpy(), *geom, b.numpy(), res.numpy(), True)
    else:
        res = None
        yr = oracle.conv2d(vr, ir, s.kh, s.kw, s.c_in, s.tile_t, x.numpy(), *geom, b.numpy(), False)
    ys = [nm.nm_conv2d(hnd, x.cuda(), s.kh, s.kw, s.stride, s.pad, s.dil, b.cuda(), residual, plan=plan,
                       residual=res.cuda() if residual else None) for _ in range(12)]
    nm.nm_weights_check(hnd)
    for y in ys:
        assert np.array_equal(y.cpu().numpy(), yr)


def test_activations_are_rounded_to_nearest():
    """A value half a TF32 step above a representable one rounds away from zero (a truncating operand would keep it below)."""
    from paper_2507_17301_b200 import nm
    x = torch.full((1, 4, 4, 4), 1.0 + 2.0 ** -11, device="cuda")
    hnd = nm.nm_prune(torch.ones((4, 1, 1, 4), device="cuda"), 4, 4, 4)
    plan = nm.nm_plan_t()
    plan.variant = 1
    y = nm.nm_conv2d(hnd, x, 1, 1, plan=plan)
    assert torch.equal(y, torch.full_like(y, 4.0 * (1.0 + 2.0 ** -10)))


def test_pruned_columns_are_never_read():
    from paper_2507_17301_b200 import nm
    x = torch.randn((2, 9, 9, 10), device="cuda")
    w = torch.randn((8, 3, 3, 10), device="cuda")
    w[..., 4] = 0.0                                   # channel 4 loses in every group of five
    hnd = nm.nm_prune(w, 2, 5, 8)
    plan = nm.nm_plan_t()
    plan.variant = 1
    y = nm.nm_conv2d(hnd, x, 3, 3, 1, 1, 1, plan=plan)
    x[..., 4] = float("inf")
    assert torch.equal(nm.nm_conv2d(hnd, x, 3, 3, 1, 1, 1, plan=plan), y)


@pytest.mark.parametrize("batch", [4, 5])                # 1280 and 1600 units of a block, tile and chunk: the gather, runs of rows
def test_default_on_both_sides_of_the_row_runs(batch):
    from paper_2507_17301_b200 import nm
    s = ConvShape("rows", batch, 49, 52, 24, 56, 3, 3, 1, 1, 1, 2, 4, 16)
    w, x, b = inputs.make_int_case(s)
    vr, ir = oracle.prune(w.numpy(), 2, 4, 16)
    yr = oracle.conv2d(vr, ir, 3, 3, 24, 16, x.numpy(), (1, 1), (1, 1), (1, 1), b.numpy(), True)
    hnd = nm.nm_prune(w.cuda(), 2, 4, 16)
    y = nm.nm_conv2d(hnd, x.cuda(), 3, 3, 1, 1, 1, b.cuda(), True)
    nm.nm_weights_check(hnd)
    assert np.array_equal(y.cpu().numpy(), yr)


@pytest.mark.parametrize("s", [
    ConvShape("tma", 4, 56, 56, 64, 64, 1, 1, 1, 0, 1, 2, 4, 8),            # the slab kernel: 98 blocks of 8 tiles, one chunk
    ConvShape("tma_tail", 3, 57, 55, 32, 76, 3, 3, 1, 1, 1, 1, 8, 8),       # last tile of four channels, last block ragged
    ConvShape("no_tma", 2, 40, 40, 36, 60, 1, 1, 1, 0, 1, 2, 4, 2),         # channels and tile width that no tensor map takes
    ConvShape("many_chunks", 1, 56, 56, 96, 200, 3, 3, 1, 1, 1, 2, 4, 8),   # the gather kernel: 14 chunks
], ids=lambda s: s.name)
def test_default_for_many_narrow_tiles(s):
    from paper_2507_17301_b200 import nm
    w, x, b = inputs.make_int_case(s)
    vr, ir = oracle.prune(w.numpy(), s.n_keep, s.m_group, s.tile_t)
    yr = oracle.conv2d(vr, ir, s.kh, s.kw, s.c_in, s.tile_t, x.numpy(), (1, 1), (s.pad,) * 2, (1, 1), b.numpy(), True)
    hnd = nm.nm_prune(w.cuda(), s.n_keep, s.m_group, s.tile_t)
    y = nm.nm_conv2d(hnd, x.cuda(), s.kh, s.kw, 1, s.pad, 1, b.cuda(), True)
    nm.nm_weights_check(hnd)
    assert np.array_equal(y.cpu().numpy(), yr)
