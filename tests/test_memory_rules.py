"""Rules of the library's code that need no device, compiled here for the host: which memory the handle-building kernels may
touch, and what the self-checking build lets an access pass by."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


def _run(tmp_path, body):
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text('#include <cstdio>\n#include "nm_internal.h"\nint main()\n{\n' + body + "}\n")
    subprocess.check_call(["g++", "-std=c++17", f"-I{ROOT}/paper_2507_17301_b200/csrc", f"-I{CUDA}/include", "-o", str(exe), str(src)])
    return subprocess.check_output([str(exe)], text=True)


def test_kernels_touch_memory_of_their_own_device_only(tmp_path):
    """Export from a handle of another GPU, and import of arrays that lie there, go through copies."""
    out = _run(tmp_path,
               "    for (cudaMemoryType t : {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice, cudaMemoryTypeManaged})\n"
               "        for (int owner : {-2, 0, 1})\n"
               '            for (int current : {0, 1}) std::printf("%d", nmhost::kernel_may_touch(t, owner, current) ? 1 : 0);\n')
    assert out == "000000" + "000000" + "001001" + "111111"     # unregistered, pinned, device (own device only), managed


def test_what_the_self_checking_build_lets_pass(tmp_path):
    out = _run(tmp_path,
               "    for (uint32_t tap : {0u, (2u << 24) | (1u << 16) | 7u, 3u << 24, 2u << 16, 8u, 0xFFFFFFFFu})\n"
               '        std::printf("%d", nm_tap_in_layer(tap, 3, 2, 8) ? 1 : 0);\n'
               '    std::printf(" ");\n'
               "    for (uint64_t at : {99ull, 100ull, 196ull, 197ull, 200ull, 0xFFFFFFFFull})\n"
               '        std::printf("%d", nm_bytes_in_span(at, 4, 100, 200) ? 1 : 0);\n')
    assert out == "110000 011000"


def test_no_check_of_the_self_checking_build_guards_an_empty_statement():
    """A check that is not part of the access's condition records a bad address and reads it all the same."""
    for name in os.listdir(f"{ROOT}/paper_2507_17301_b200/csrc"):
        with open(f"{ROOT}/paper_2507_17301_b200/csrc/{name}") as f:
            assert not re.search(r"NM_CHECKED\([^;{]*\)\s*\{\s*\}", f.read()), name


def test_shared_arrays_read_as_vectors_are_aligned_for_them():
    """A float array may start at any multiple of four bytes; read as float4 it has to say that it does not."""
    vectors = {"float4": 16, "uint4": 16, "int4": 16, "double2": 16, "float2": 8, "uint2": 8, "int2": 8}
    found = 0
    for name in os.listdir(f"{ROOT}/paper_2507_17301_b200/csrc"):
        with open(f"{ROOT}/paper_2507_17301_b200/csrc/{name}") as f:
            text = f.read()
        for align, arrays in re.findall(r"__shared__\s+(?:__align__\((\d+)\)\s+)?(?:float|int|uint32_t|uint16_t|uint8_t|short)\s+([^;]*);", text):
            for array in re.findall(r"(\w+)\[", arrays):
                for vector in re.findall(rf"reinterpret_cast<(?:const )?(\w+)\s*\*>\(&?{array}\b", text):
                    if vector in vectors:
                        found += 1
                        assert int(align or 4) >= vectors[vector], (name, array, vector)
    assert found >= 2


def test_which_pointwise_layers_read_more_than_they_write(tmp_path):
    """A strided layer reads the pixels it computes from, not its whole input: 256 -> 512 by 2 reads half of what it writes."""
    out = _run(tmp_path,
               "    for (int stride : {1, 2})\n"
               "        for (int c_out : {128, 256, 512}) {\n"
               "            ConvParams p = {};\n"
               "            p.batch = 2; p.h = p.w = 56; p.c_in = 256; p.c_out = c_out; p.stride_h = p.stride_w = stride;\n"
               "            p.ho = p.wo = (56 + stride - 1) / stride; p.pixels = 2ll * p.ho * p.wo;\n"
               '            std::printf("%d", nm_pointwise_reads_more(p) ? 1 : 0);\n'
               "        }\n")
    assert out == "100100"
