"""The per-call extension: argument checks (no GPU) and the output it allocates."""
import ctypes
import os
import subprocess
import sys

import pytest
import torch

from paper_2507_17301_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

build.build()
from paper_2507_17301_b200 import nm  # noqa: E402


def test_host_tensors_and_wrong_types_are_refused():
    x = torch.zeros(1, 4, 4, 8)
    w = nm.Weights.__new__(nm.Weights)
    w._h, w._addr, w.c_out = None, 0, 8
    for bad in (x, x.double(), None, 3):
        with pytest.raises(TypeError, match="x must be a contiguous float32 CUDA tensor"):
            nm.nm_conv2d(w, bad, 1, 1)
        with pytest.raises(TypeError, match="x must be"):
            nm.nm_maxpool2d(bad)
    with pytest.raises((TypeError, IndexError)):
        nm.nm_conv2d(w, x, 1, 1, stride=(1,))


def test_a_plan_of_another_type_is_refused():
    w = nm.Weights.__new__(nm.Weights)
    w._h, w._addr, w.c_out = None, 0, 8
    x = torch.zeros(1, 4, 4, 8)
    for bad in (ctypes.c_int(4), (ctypes.c_int * 16)(), nm.nm_plan_t):
        with pytest.raises((ctypes.ArgumentError, TypeError), match="plan|ctypes|invalid type"):
            nm.nm_conv2d(w, x, 1, 1, plan=bad)
    with pytest.raises(TypeError, match="x must be"):       # the plan is looked at first and is in order
        nm.nm_conv2d(w, x, 1, 1, plan=nm.nm_plan_t())


@pytest.mark.gpu
def test_the_window_is_not_needed_beside_an_output():
    x = torch.randn(1, 5, 5, 8, device="cuda")
    hnd = nm.nm_prune(torch.randn(12, 3, 3, 8, device="cuda"), 2, 4, 4)
    y = nm.nm_conv2d(hnd, x, 3, 3, 1, 1)
    assert torch.equal(nm.nm_conv2d(hnd, x, None, None, 1, 1, y=torch.empty_like(y)), y)


def test_no_usable_device_is_a_python_exception():
    """In a process of its own: a C++ exception that leaves the extension ends the process."""
    code = ("from paper_2507_17301_b200 import nm\n"
            "try:\n    nm._stream()\nexcept RuntimeError:\n    print('refused')\n")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, CUDA_VISIBLE_DEVICES=""), capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "refused", r.stderr[-1000:]


@pytest.mark.gpu
@pytest.mark.parametrize("h,w,k,stride,pad,dil", [(7, 9, 3, (2, 1), (1, 0), (1, 2)), (5, 5, 5, 1, 0, 1), (8, 3, 1, 3, 0, 1)])
def test_allocated_output_has_the_librarys_shape(h, w, k, stride, pad, dil):
    x = torch.randn(2, h, w, 8, device="cuda")
    hnd = nm.nm_prune(torch.randn(12, k, k, 8, device="cuda"), 2, 4, 4)
    y = nm.nm_conv2d(hnd, x, k, k, stride, pad, dil)
    assert tuple(y.shape) == nm.out_shape(x.shape, k, k, 12, nm._pair(stride), nm._pair(pad), nm._pair(dil))
    given = torch.empty_like(y)
    assert nm.nm_conv2d(hnd, x, k, k, stride, pad, dil, y=given) is given
    assert torch.equal(given, y)
    with pytest.raises(TypeError, match="residual must have the output's shape"):
        nm.nm_conv2d(hnd, x, k, k, stride, pad, dil, residual=torch.zeros(1, 1, 1, 12, device="cuda"))
    with pytest.raises(TypeError, match="y must be"):
        nm.nm_conv2d(hnd, x, k, k, stride, pad, dil, y=given.double())
    hnd.free()
    with pytest.raises(nm.NmError):
        nm.nm_conv2d(hnd, x, k, k, stride, pad, dil)


@pytest.mark.gpu
def test_calls_go_to_the_current_stream():
    x = torch.randn(1, 6, 6, 8, device="cuda")
    side = torch.cuda.Stream()
    assert nm._stream() == torch.cuda.current_stream().cuda_stream
    with torch.cuda.stream(side):
        assert nm._stream() == side.cuda_stream
    assert torch.equal(nm.nm_maxpool2d(x, 2, 2, 0), torch.nn.functional.max_pool2d(x.permute(0, 3, 1, 2), 2, 2).permute(0, 2, 3, 1))
