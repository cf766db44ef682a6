"""The one-launch pruning pass at the edges of its blocks (spans of whole groups, 128 columns at most; wider groups take
the three-kernel form), and handles built on memory that an earlier handle used."""
import numpy as np
import pytest
import torch

import oracle
from parity import assert_prune_bit_exact

pytestmark = pytest.mark.gpu


def _check(w, n, m, t):
    from paper_2507_17301_b200 import nm
    hnd = nm.nm_prune(w.cuda(), n, m, t)
    v, i = nm.nm_weights_export(hnd)
    vr, ir = oracle.prune(w.numpy(), n, m, t)
    assert_prune_bit_exact(v.cpu().numpy(), i.cpu().numpy(), vr, ir)
    return hnd


@pytest.mark.parametrize("n,m", [(1, 1), (1, 3), (2, 5), (60, 127), (64, 128), (65, 129), (3, 200)])
@pytest.mark.parametrize("t,c_out,k", [(16, 33, 127), (17, 40, 128), (1, 3, 129), (256, 300, 385)])
def test_span_edges(n, m, t, c_out, k):
    g = torch.Generator().manual_seed(m * 1000 + k)
    _check(torch.randint(-3, 4, (c_out, 1, 1, k), generator=g).float(), n, m, t)   # few distinct scores: ties too


def test_memory_of_a_freed_handle_leaves_nothing_behind():
    """The second handle takes the first one's block: its convolution is the one a fresh handle gives."""
    from paper_2507_17301_b200 import nm
    g = torch.Generator().manual_seed(1)
    x = torch.randn((1, 9, 9, 64), generator=g).cuda()
    for n, m, t in ((4, 4, 16), (1, 8, 16), (3, 4, 24), (2, 4, 16)):
        for _ in range(2):
            w = torch.randn((40, 3, 3, 64), generator=g)
            hnd = _check(w, n, m, t)
            y = nm.nm_conv2d(hnd, x, 3, 3, 1, 1, 1)
            vr, ir = oracle.prune(w.numpy(), n, m, t)
            yr = oracle.conv2d(vr, ir, 3, 3, 64, t, x.cpu().numpy(), (1, 1), (1, 1), (1, 1), None, False)
            assert np.linalg.norm(y.cpu().numpy() - yr) <= 2e-3 * np.linalg.norm(yr)   # TF32 operands, as in parity.py
            hnd.free()
