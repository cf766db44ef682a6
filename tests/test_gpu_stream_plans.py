"""What a plan can ask of the stream kernel: every group of tiles that the library default may take, whether or not it divides the layer's
tiles, and nothing the kernel cannot hold; and the tuner times the group that a call without a plan takes."""
import numpy as np
import pytest
import torch

import oracle
from paper_2507_17301_b200.inputs import ConvShape
from parity import oracle_layer, tensors_for

pytestmark = pytest.mark.gpu

# shape, groups (tiles per CTA) that whole blocks of 32 channels and 256 of them admit
SHAPES = [
    (ConvShape("five_tiles", 3, 31, 37, 96, 80, 3, 3, 2, 2, 2, 3, 4, 16), {2, 4}),
    (ConvShape("three_of_48", 4, 30, 30, 96, 144, 1, 1, 1, 0, 1, 2, 4, 48), {2, 4}),
    (ConvShape("five_of_32", 2, 33, 31, 64, 160, 1, 1, 1, 0, 1, 1, 4, 32), {1, 2, 3, 4}),
    (ConvShape("one_of_16", 8, 40, 33, 32, 16, 3, 3, 1, 1, 1, 2, 8, 16), {2, 4}),
    (ConvShape("three_of_128", 2, 28, 28, 64, 384, 1, 1, 1, 0, 1, 2, 4, 128), {1, 2}),
]


@pytest.mark.parametrize("residual", [False, True])
@pytest.mark.parametrize("s,groups", SHAPES, ids=lambda v: getattr(v, "name", None))
def test_groups_that_need_not_divide_the_tiles(s, groups, residual):
    from paper_2507_17301_b200 import nm
    w, x, b = tensors_for(s, True)
    values, indices, yr = oracle_layer(s, w, x, b)
    r = None
    if residual:
        r = torch.randint(-4, 5, yr.shape, generator=torch.Generator().manual_seed(5)).float()
        yr = oracle.conv2d_res(values, indices, s.kh, s.kw, s.c_in, s.tile_t, x.numpy(), (s.stride,) * 2, (s.pad,) * 2, (s.dil,) * 2, b.numpy(),
                               r.numpy(), s.relu)
    hnd = nm.nm_prune(w.cuda(), s.n_keep, s.m_group, s.tile_t)
    ran = set()
    for group in range(0, 6):
        p = nm.nm_plan_t()
        p.variant, p.bn = 3, group * s.tile_t
        y = torch.full(yr.shape, float("nan"), device="cuda")
        try:
            nm.nm_conv2d(hnd, x.cuda(), s.kh, s.kw, s.stride, s.pad, s.dil, b.cuda(), s.relu, y, p, r.cuda() if residual else None)
        except nm.NmError as e:
            assert e.status == nm.NM_ERR_UNSUPPORTED
            continue
        nm.nm_weights_check(hnd)
        ran.add(group)
        assert np.array_equal(y.cpu().numpy(), yr), group
    assert ran == groups | {0}      # (0: the library's choice)


def test_tuner_lists_the_group_of_a_call_without_a_plan(monkeypatch):
    from paper_2507_17301_b200 import nm
    monkeypatch.setenv("NM_AUTOTUNE_VARIANTS", "3")
    s = SHAPES[0][0]
    w, x, b = (t.cuda() for t in tensors_for(s))
    hnd = nm.nm_prune(w, s.n_keep, s.m_group, s.tile_t)
    plan = nm.nm_autotune(hnd, x, s.stride, s.pad, s.dil, b, s.relu, None, s.kh, s.kw)[0]
    assert plan.variant == 3
