"""Order of the additions at the end of a layer, bit for bit: sum over the columns, then bias, then shortcut; the kernels of
SHORTCUT_FIRST add bias + shortcut to the sum.  A network of many layers that truncate their inputs carries a last bit that moved into
its fourth digit."""
import pytest
import torch

from paper_2507_17301_b200.inputs import ConvShape
from parity import tensors_for
from test_gpu_conv import _plans

pytestmark = pytest.mark.gpu

SHORTCUT_FIRST = (2, 5, 6, 10)   # the slab kernel (2) for whole blocks of 32 channels

SHAPES = [
    (ConvShape("pointwise", 4, 28, 28, 128, 256, 1, 1, 1, 0, 1, 2, 4, 64), {1, 2, 3, 4, 7, 8, 10}),
    (ConvShape("pw_few_channels", 2, 56, 56, 24, 144, 1, 1, 1, 0, 1, 2, 4, 16), {1, 2, 4}),
    (ConvShape("3x3", 4, 14, 14, 256, 256, 3, 3, 1, 1, 1, 2, 8, 32), {1, 2, 3, 4, 6, 8, 10}),
    (ConvShape("strided", 2, 29, 31, 64, 128, 3, 3, 2, 1, 1, 2, 4, 32), {1, 2, 3, 4}),
    (ConvShape("few_channels", 2, 32, 32, 3, 64, 7, 7, 2, 3, 1, 1, 1, 64), {1, 2, 5, 9}),
]


def _all_plans(nm, s):
    plans = [p for p in _plans(nm, s) if p is not None]
    for split, kblk, issuers in ((2, 0, 0), (3, 2, 0), (2, 0, 2), (-1, 0, 0), (-1, 2, 2)):
        p = nm.nm_plan_t()
        p.variant, p.bn, p.split, p.kblk, p.issuers = 4, 64, split, kblk, issuers
        plans.append(p)
    for variant, ksplits in ((8, (1, 2, 3)), (10, (1, 2, 4, 8))):
        for ksplit in ksplits:
            p = nm.nm_plan_t()
            p.variant, p.bn, p.ksplit = variant, 64, ksplit
            plans.append(p)
    return plans


@pytest.mark.parametrize("s,variants", SHAPES, ids=lambda v: getattr(v, "name", ""))
def test_bias_then_shortcut(s, variants):
    from paper_2507_17301_b200 import nm
    w, x, b = (t.cuda() for t in tensors_for(s))
    r = torch.randn((s.batch, s.ho, s.wo, s.c_out), generator=torch.Generator().manual_seed(7)).cuda()
    hnd = nm.nm_prune(w, s.n_keep, s.m_group, s.tile_t)
    plans = _all_plans(nm, s)
    shape = (s.batch, s.h, s.w, s.c_in)
    nm.nm_weights_reserve(hnd, max(nm.nm_plan_scratch_bytes(hnd, shape, s.stride, s.pad, s.dil, p) for p in plans))
    ran = set()
    for plan in plans:
        try:
            acc = nm.nm_conv2d(hnd, x, s.kh, s.kw, s.stride, s.pad, s.dil, None, False, plan=plan)
            y = nm.nm_conv2d(hnd, x, s.kh, s.kw, s.stride, s.pad, s.dil, b, True, plan=plan, residual=r)
        except nm.NmError as e:
            assert e.status == nm.NM_ERR_UNSUPPORTED
            continue
        nm.nm_weights_check(hnd)
        ran.add(plan.variant)
        first = plan.variant in SHORTCUT_FIRST and (plan.variant != 2 or s.tile_t % 32 == 0)
        assert torch.equal(y, torch.relu(acc + (b + r) if first else (acc + b) + r)), plan.as_dict()
    assert variants <= ran, (variants, ran)
