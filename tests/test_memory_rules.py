"""Which memory the handle-building kernels may touch: a rule of the host code, compiled here without a device."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


def test_kernels_touch_memory_of_their_own_device_only(tmp_path):
    """Export from a handle of another GPU, and import of arrays that lie there, go through copies."""
    src = tmp_path / "rule.cpp"
    src.write_text('#include <cstdio>\n#include "nm_internal.h"\nint main()\n{\n'
                   "    for (cudaMemoryType t : {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice, cudaMemoryTypeManaged})\n"
                   "        for (int owner : {-2, 0, 1})\n"
                   '            for (int current : {0, 1}) std::printf("%d", nmhost::kernel_may_touch(t, owner, current) ? 1 : 0);\n}\n')
    exe = tmp_path / "rule"
    subprocess.check_call(["g++", "-std=c++17", f"-I{ROOT}/paper_2507_17301_b200/csrc", f"-I{CUDA}/include", "-o", str(exe), str(src)])
    out = subprocess.check_output([str(exe)], text=True)
    assert out == "000000" + "000000" + "001001" + "111111"     # unregistered, pinned, device (own device only), managed
