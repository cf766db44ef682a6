"""The kernel that builds a handle: rows of a tile dealt to several blocks, columns and rows that end inside a 32-column block or a span, the
same layouts from dense weights and from the compressed form, and more creating calls at once than there are slots for their sums."""
import threading
import time

import numpy as np
import pytest
import torch

import oracle
from parity import assert_prune_bit_exact

pytestmark = pytest.mark.gpu

# c_out, kh, kw, c_in, N, M, T
SHAPES = [
    (72, 1, 1, 100, 2, 4, 72),      # two blocks of rows, the second of 8; K ends inside a 32-column block, c_out too
    (200, 3, 3, 32, 3, 4, 200),     # four blocks of rows; the last span holds 32 of its columns
    (96, 3, 3, 64, 2, 8, 32),       # select layout, four steps to a chunk
    (64, 1, 1, 128, 1, 8, 64),      # select layout with steps of 64 columns
    (68, 1, 1, 63, 1, 3, 16),       # spans of 126 columns; a tail group; a last tile of 4 rows
    (32, 7, 7, 3, 1, 1, 32),        # plane layout
    # groups wider than a block: selected and laid out by kernels of their own
    (64, 1, 1, 256, 256, 256, 32),  # slab layout (everything kept)
    (32, 7, 7, 3, 100, 147, 32),    # plane layout with zeros
    (100, 3, 3, 64, 100, 192, 48),  # expanded layout with zeros; a last tile of 4 rows
]


@pytest.mark.parametrize("c_out,kh,kw,c_in,n,m,t", SHAPES)
def test_layouts_from_dense_weights_and_from_the_compressed_form(c_out, kh, kw, c_in, n, m, t):
    from paper_2507_17301_b200 import nm
    g = torch.Generator().manual_seed(c_out + c_in)
    w = torch.randint(-4, 5, (c_out, kh, kw, c_in), generator=g).float()
    x = torch.randint(-4, 5, (4, 17, 19, c_in), generator=g).float()
    pruned = nm.nm_prune(w.cuda(), n, m, t)
    v, i = nm.nm_weights_export(pruned)
    vr, ir = oracle.prune(w.numpy(), n, m, t)
    assert_prune_bit_exact(v.cpu().numpy(), i.cpu().numpy(), vr, ir)
    kept, total = nm.nm_weights_retained_l1(pruned)
    assert (kept, total) == (float(np.abs(vr.astype(np.float64)).sum()), float(w.double().abs().sum()))   # integers: exact in any order
    imported = nm.nm_weights_import(v, i, kh, kw, c_in, n, m, t)
    v2, i2 = nm.nm_weights_export(imported)
    assert torch.equal(v, v2) and torch.equal(i.view(torch.int16), i2.view(torch.int16))
    yr = oracle.conv2d(vr, ir, kh, kw, c_in, t, x.numpy(), (1, 1), (kh // 2, kw // 2), (1, 1), None, False)
    ran = 0
    for variant in range(1, 11):
        plan = nm.nm_plan_t()
        plan.variant = variant
        for hnd in (pruned, imported):
            try:
                y = nm.nm_conv2d(hnd, x.cuda(), kh, kw, 1, (kh // 2, kw // 2), 1, plan=plan)
            except nm.NmError as e:
                assert e.status == nm.NM_ERR_UNSUPPORTED
                continue
            nm.nm_weights_check(hnd)
            ran += 1
            assert np.array_equal(y.cpu().numpy(), yr), variant
    assert ran >= 2   # the gather kernel takes every shape


def test_more_creating_calls_at_once_than_slots():
    """48 calls, each behind a kernel that spins for a while on its stream: at least 33 have launched their own kernel before the first returns, so one at
    least has no slot for its sums."""
    from paper_2507_17301_b200 import nm
    weights = [torch.randint(-4, 5, (48, 3, 3, 32), generator=torch.Generator().manual_seed(s)).float().cuda() for s in range(48)]
    blocks = [nm.nm_prune(w, 2, 4, 16) for w in weights]
    del blocks                              # (their memory is kept and taken again: no allocation waits for the spinning kernels)
    torch.cuda.synchronize()
    handles = [None] * len(weights)
    go = threading.Barrier(len(weights))

    def create(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            go.wait()
            torch.cuda._sleep(1_000_000_000)   # half a second
            handles[i] = nm.nm_prune(weights[i], 2, 4, 16)

    threads = [threading.Thread(target=create, args=(i,)) for i in range(len(weights))]
    launched = nm.nm_launch_count()
    for th in threads:
        th.start()
    in_flight, deadline = 0, time.monotonic() + 30
    while in_flight <= 32 and any(th.is_alive() for th in threads) and time.monotonic() < deadline:
        count = nm.nm_launch_count() - launched                # (before the calls that have returned are counted: never too many)
        in_flight = max(in_flight, count - sum(hnd is not None for hnd in handles))
        time.sleep(1e-3)
    for th in threads:
        th.join()
    assert in_flight > 32, in_flight
    for w, hnd in zip(weights, handles):
        kept, total = nm.nm_weights_retained_l1(hnd)
        assert kept == nm.nm_weights_export(hnd)[0].double().abs().sum().item() and total == w.double().abs().sum().item()
