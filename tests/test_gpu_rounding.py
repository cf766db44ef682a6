"""Activations are rounded to TF32 to nearest by the kernels that say so: inputs rounded beforehand give the very same output,
bit for bit.  Those are the compacting ones (ties away from zero, cvt.rna) and the cluster kernel for inputs below 128 KiB,
which no other kernel of the tuner truncates (tensor maps of type TFLOAT32, ties to even); a truncating operand fails either way."""
import pytest
import torch

from paper_2507_17301_b200.inputs import ConvShape
from parity import tensors_for

pytestmark = pytest.mark.gpu

C3 = ConvShape("3x3", 2, 28, 28, 64, 128, 3, 3, 1, 1, 1, 2, 4, 32)
C1 = ConvShape("1x1", 2, 28, 28, 128, 256, 1, 1, 1, 0, 1, 2, 4, 64)
S2 = ConvShape("3x3_s2", 2, 28, 28, 64, 64, 3, 3, 2, 1, 1, 1, 4, 16)
BOX = ConvShape("7x7_map", 1, 7, 7, 128, 64, 3, 3, 1, 1, 1, 2, 4, 32)        # below 128 KiB
ROWS = ConvShape("7x7_rows", 1, 7, 7, 512, 96, 1, 1, 1, 0, 1, 2, 8, 8)      # below 128 KiB
ODD = ConvShape("odd", 2, 17, 15, 20, 64, 3, 3, 1, 1, 1, 2, 4, 8)

CASES = [
    (1, {}, C3, "away"), (1, {}, ODD, "away"), (2, {}, C3, "away"), (2, {"split": 1}, ODD, "away"), (3, {}, C1, "away"), (3, {}, S2, "away"),
    (10, {"bn": 64, "ksplit": 8}, BOX, "even"), (10, {"bn": 32, "ksplit": 4, "stages": 2}, ROWS, "even"),
]


def round_tf32(x, ties):
    bits = x.view(torch.int32)
    up = 0x1000 if ties == "away" else 0xFFF + ((bits >> 13) & 1)
    return ((bits + up) & ~0x1FFF).view(torch.float32)


@pytest.mark.parametrize("variant,fields,s,ties", CASES, ids=lambda v: getattr(v, "name", None) or str(v).replace(" ", ""))
def test_activations_are_rounded_to_nearest(variant, fields, s, ties):
    from paper_2507_17301_b200 import nm
    w, x, b = (t.cuda() for t in tensors_for(s))
    bits = x.view(torch.int32)
    bits.view(-1)[::3] = (bits.view(-1)[::3] & ~0x1FFF) | 0x1000      # every third value half-way between two neighbours
    hnd = nm.nm_prune(w, s.n_keep, s.m_group, s.tile_t)
    plan = nm.nm_plan_t()
    plan.variant = variant
    for name, value in fields.items():
        setattr(plan, name, value)
    y, y_tf32 = (nm.nm_conv2d(hnd, v, s.kh, s.kw, s.stride, s.pad, s.dil, b, plan=plan) for v in (x, round_tf32(x, ties)))
    nm.nm_weights_check(hnd)
    assert torch.equal(y, y_tf32)
