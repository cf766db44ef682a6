"""The stream kernel's rings against the CPU oracle, bit for bit on integer inputs: one and two compactor teams, rings of odd and even depth that
come round several times, one and two staging boxes, several items per CTA with an odd number of chunks each (so that the teams'
chunks change from item to item)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2507_17301_b200.inputs import ConvShape
from parity import oracle_layer, tensors_for

pytestmark = pytest.mark.gpu

# shape, tiles per CTA, depths that fit (by the layer's bytes per stage); more than 148 pixel blocks x groups, i.e. several items for a CTA
SHAPES = [
    (ConvShape("two_teams_27_chunks", 8, 56, 56, 96, 128, 3, 3, 1, 1, 1, 3, 4, 32), 2, {1, 2, 3, 4, 5, 6}),     # 864 columns, 32 at a time; 392 items
    (ConvShape("two_teams_9_chunks", 6, 56, 56, 64, 128, 3, 3, 1, 1, 1, 2, 4, 64), 1, {1, 2, 3, 4, 5}),         # 576 columns, 64 at a time; five with one box
    (ConvShape("two_teams_wide_stage", 4, 50, 50, 64, 384, 3, 3, 1, 1, 1, 2, 8, 96), 2, {1, 2, 3}),             # 192 channels and one accumulator
    (ConvShape("one_team_9_chunks", 6, 56, 56, 64, 64, 3, 3, 1, 1, 1, 1, 8, 32), 1, {1, 2, 3, 4, 5}),           # eight kept columns of a chunk
    (ConvShape("one_team_one_chunk", 8, 56, 56, 64, 256, 1, 1, 1, 0, 1, 2, 4, 64), 1, {1, 2, 3, 4, 5}),
]


@pytest.mark.parametrize("residual", [False, True])
@pytest.mark.parametrize("s,tiles,depths", SHAPES, ids=lambda v: getattr(v, "name", None))
def test_every_depth_integer_exact(s, tiles, depths, residual):
    from paper_2507_17301_b200 import nm
    w, x, b = tensors_for(s, True)
    values, indices, yr = oracle_layer(s, w, x, b)
    r = None
    if residual:
        r = torch.randint(-4, 5, yr.shape, generator=torch.Generator().manual_seed(5)).float()
        yr = oracle.conv2d_res(values, indices, s.kh, s.kw, s.c_in, s.tile_t, x.numpy(), (s.stride,) * 2, (s.pad,) * 2, (s.dil,) * 2, b.numpy(),
                               r.numpy(), s.relu)
    hnd = nm.nm_prune(w.cuda(), s.n_keep, s.m_group, s.tile_t)
    xd, bd, rd = x.cuda(), b.cuda(), r.cuda() if residual else None
    ran = set()
    for stages in range(0, 8):
        p = nm.nm_plan_t()
        p.variant, p.bn, p.stages = 3, tiles * s.tile_t, stages
        y = torch.full(yr.shape, float("nan"), device="cuda")
        try:
            nm.nm_conv2d(hnd, xd, s.kh, s.kw, s.stride, s.pad, s.dil, bd, s.relu, y, p, rd)
        except nm.NmError as e:
            assert e.status == nm.NM_ERR_UNSUPPORTED
            continue
        nm.nm_weights_check(hnd)
        ran.add(stages)
        assert np.array_equal(y.cpu().numpy(), yr), stages
    assert ran == depths | {0}
