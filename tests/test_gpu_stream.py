"""The stream kernel against the CPU oracle, bit for bit on integer inputs: tiles dealt out in groups that do not divide them (library default, which
has to take the kernel here, and plans), one to three chunks, shallow and deep rings, several items per CTA, the fused shortcut."""
import numpy as np
import pytest
import torch

import oracle
from paper_2507_17301_b200.inputs import ConvShape
from parity import kernels_of, oracle_layer, tensors_for

pytestmark = pytest.mark.gpu

# shape, widths a plan can ask for (0: the library's choice; one tile and two), depths that fit all of them
SHAPES = [
    (ConvShape("five_tiles", 5, 61, 75, 96, 80, 3, 3, 2, 2, 2, 3, 4, 16), (0, 2), (0, 1, 2, 3, 4, 6)),         # groups of two tiles, the last of one: 16 channels
    (ConvShape("three_tiles", 6, 40, 33, 32, 48, 3, 3, 1, 1, 1, 2, 4, 16), (0, 2), (0, 1, 2, 3, 4)),           # two groups; ragged last pixel block
    (ConvShape("many_items", 8, 56, 56, 32, 112, 1, 1, 1, 0, 1, 2, 4, 16), (0, 2), (0, 1, 2, 3, 4)),           # one chunk
    (ConvShape("two_chunks", 8, 30, 30, 128, 96, 1, 1, 1, 0, 1, 1, 8, 32), (0, 1, 2), (0, 1, 2, 3, 4)),
    (ConvShape("three_chunks", 4, 30, 30, 96, 144, 1, 1, 1, 0, 1, 3, 4, 48), (0, 2), (0, 1, 2, 3, 4, 6)),      # tiles of 48 channels, grouped by two
    (ConvShape("dense_odd", 2, 33, 31, 64, 160, 1, 1, 1, 0, 1, 4, 4, 32), (0, 1, 2), (0, 1, 2, 3, 4, 6)),
]


@pytest.mark.parametrize("residual", [False, True])
@pytest.mark.parametrize("s,widths,depths", SHAPES, ids=lambda v: getattr(v, "name", ""))
def test_default_and_plans_integer_exact(s, widths, depths, residual):
    from paper_2507_17301_b200 import nm
    w, x, b = tensors_for(s, True)
    values, indices, yr = oracle_layer(s, w, x, b)
    r = None
    if residual:
        r = torch.randint(-4, 5, yr.shape, generator=torch.Generator().manual_seed(5)).float()
        yr = oracle.conv2d(values, indices, s.kh, s.kw, s.c_in, s.tile_t, x.numpy(), (s.stride,) * 2, (s.pad,) * 2, (s.dil,) * 2, b.numpy(), False)
        yr = np.maximum(yr + r.numpy(), 0.0) if s.relu else yr + r.numpy()
    hnd = nm.nm_prune(w.cuda(), s.n_keep, s.m_group, s.tile_t)
    xd, bd, rd = x.cuda(), b.cuda(), r.cuda() if residual else None
    assert kernels_of(lambda: nm.nm_conv2d(hnd, xd, s.kh, s.kw, s.stride, s.pad, s.dil, bd, s.relu, residual=rd)) == ["k_conv_stream"]
    plans = {None: None}
    for width in (0, 1, 2):
        for stages in (0, 1, 2, 3, 4, 6):
            p = plans[width, stages] = nm.nm_plan_t()
            p.variant, p.bn, p.stages = 3, width * s.tile_t, stages
    ran = set()
    for key, plan in plans.items():
        y = torch.full(yr.shape, float("nan"), device="cuda")
        try:
            nm.nm_conv2d(hnd, xd, s.kh, s.kw, s.stride, s.pad, s.dil, bd, s.relu, y, plan, rd)
        except nm.NmError as e:
            assert plan is not None and e.status == nm.NM_ERR_UNSUPPORTED
            continue
        nm.nm_weights_check(hnd)
        ran.add(key)
        assert np.array_equal(y.cpu().numpy(), yr), key
    assert ran == {None} | {(width, stages) for width in widths for stages in depths}
