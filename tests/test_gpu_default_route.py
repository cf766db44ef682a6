"""Which of the gathering kernels a call without a plan runs: the stream kernel where a pixel block serves several tiles or there are many, the
gather kernel where one tile reads a block anyway, or few blocks leave SMs to split the chunks over."""
import pytest
import torch

from paper_2507_17301_b200.inputs import ConvShape
from parity import kernels_of

pytestmark = pytest.mark.gpu

ROUTES = [
    (ConvShape("one_tile_16_3x3", 23, 76, 25, 192, 16, 3, 3, 1, 1, 1, 1, 8, 16), "k_conv_gather"),
    (ConvShape("one_tile_48_5x5", 22, 21, 44, 64, 48, 5, 5, 1, 2, 1, 1, 4, 48), "k_conv_gather"),
    (ConvShape("one_tile_16_1x1", 2, 23, 41, 128, 16, 1, 1, 1, 0, 1, 2, 4, 16), "k_conv_gather"),
    (ConvShape("few_blocks_long", 4, 14, 14, 256, 256, 3, 3, 1, 1, 1, 2, 4, 64), "k_conv_gather"),
    (ConvShape("two_tiles_5x5", 2, 40, 69, 448, 64, 5, 5, 1, 2, 1, 2, 8, 32), "k_conv_gather"),
    (ConvShape("seven_tiles_of_48", 5, 9, 22, 128, 240, 3, 3, 2, 1, 1, 2, 8, 48), "k_conv_gather"),
    (ConvShape("five_tiles_of_16", 5, 61, 75, 96, 80, 3, 3, 2, 2, 2, 3, 4, 16), "k_conv_stream"),
    (ConvShape("four_tiles", 4, 28, 28, 128, 128, 1, 1, 1, 0, 1, 2, 4, 32), "k_conv_stream"),
    (ConvShape("many_blocks", 16, 56, 56, 64, 256, 1, 1, 1, 0, 1, 2, 4, 64), "k_conv_stream"),
    (ConvShape("long_and_many", 32, 14, 14, 256, 256, 3, 3, 1, 1, 1, 2, 4, 64), "k_conv_stream"),
]


@pytest.mark.parametrize("s,kernel", ROUTES, ids=lambda v: getattr(v, "name", v))
def test_default_takes(s, kernel):
    from paper_2507_17301_b200 import nm
    hnd = nm.nm_prune(torch.randn((s.c_out, s.kh, s.kw, s.c_in), device="cuda"), s.n_keep, s.m_group, s.tile_t)
    x = torch.randn((s.batch, s.h, s.w, s.c_in), device="cuda")
    assert kernels_of(lambda: nm.nm_conv2d(hnd, x, s.kh, s.kw, s.stride, s.pad, s.dil)) == [kernel]
