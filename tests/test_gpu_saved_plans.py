"""Plans that earlier forms of the expanded-operand and select kernels took, as a plan file may hold them: rings of a single slot,
more ranges of the reduction axis than the layer has chunks, activation rings that leave room for two weight slots.  Bit for
bit against the CPU oracle on integer inputs."""
import numpy as np
import pytest

from paper_2507_17301_b200.inputs import ConvShape
from parity import oracle_layer, tensors_for

pytestmark = pytest.mark.gpu

C3 = ConvShape("3x3", 2, 28, 28, 64, 128, 3, 3, 1, 1, 1, 2, 4, 32)
C1 = ConvShape("1x1", 3, 28, 27, 128, 192, 1, 1, 1, 0, 1, 2, 4, 64)
MANY = ConvShape("many_items", 8, 56, 56, 64, 64, 3, 3, 1, 1, 1, 2, 4, 64)                 # several items per CTA
ONE_CHUNK = ConvShape("one_chunk", 2, 28, 27, 128, 64, 1, 1, 1, 0, 1, 1, 8, 32)
THREE_CHUNKS = ConvShape("three_chunks", 2, 15, 15, 384, 64, 1, 1, 1, 0, 1, 1, 4, 64)
WIDE_3OF4 = ConvShape("wide_3of4", 2, 28, 28, 64, 128, 5, 5, 1, 2, 1, 3, 4, 128)
WIDE_1OF8 = ConvShape("wide_1of8", 3, 28, 28, 128, 256, 3, 3, 1, 1, 1, 1, 8, 256)
HALO_1OF8 = ConvShape("halo_1of8", 9, 7, 10, 256, 256, 3, 3, 1, 1, 1, 1, 8, 256)

CASES = ([(4, f, s) for s in (C3, C1, MANY) for f in ({"stages": 1}, {"stages": 1, "split": 1}, {"stages": 1, "kblk": 2, "split": 1}, {"stages": 1, "split": -1, "bn": 64})]
         + [(4, {"stages": 1, "split": 2, "bn": 64}, C3)]
         + [(8, {"ksplit": k}, s) for s in (ONE_CHUNK, THREE_CHUNKS) for k in (2, 4)]
         + [(8, {"ksplit": 8, "loads": 1}, THREE_CHUNKS), (8, {"stages": 3}, WIDE_3OF4), (8, {"stages": 4, "loads": 1}, WIDE_1OF8), (8, {"stages": 4}, HALO_1OF8)])


@pytest.mark.parametrize("variant,fields,s", CASES, ids=lambda v: getattr(v, "name", None) or str(v).replace(" ", ""))
def test_plan_is_taken_and_exact(variant, fields, s):
    from paper_2507_17301_b200 import nm
    w, x, b = tensors_for(s, True)
    _, _, yr = oracle_layer(s, w, x, b)
    hnd = nm.nm_prune(w.cuda(), s.n_keep, s.m_group, s.tile_t)
    plan = nm.nm_plan_t()
    plan.variant = variant
    for name, value in fields.items():
        setattr(plan, name, value)
    nm.nm_weights_reserve(hnd, nm.nm_plan_scratch_bytes(hnd, x.shape, s.stride, s.pad, s.dil, plan))
    ys = [nm.nm_conv2d(hnd, x.cuda(), s.kh, s.kw, s.stride, s.pad, s.dil, b.cuda(), s.relu, plan=plan) for _ in range(4)]
    nm.nm_weights_check(hnd)
    for y in ys:
        assert np.array_equal(y.cpu().numpy(), yr)
