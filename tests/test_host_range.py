"""The decision whether w4a8_linear_host's kernels use a host buffer in place, compiled for the CPU with the answers of the
driver given: the buffer has to lie within one pinned range as a whole."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_12932_b200", "csrc")


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    d = tmp_path_factory.mktemp("host_range")
    (d / "shim.cpp").write_text('#include "host_range.h"\n'
                                'extern "C" uint64_t in_place(int pinned, uint64_t device, uint64_t start, uint64_t size, uint64_t p, uint64_t bytes) {\n'
                                '    const w4a8::HostMemory m = {pinned != 0, (void*)device, start, size};\n'
                                '    return (uint64_t)w4a8::in_place_address(m, (const void*)p, bytes);\n}\n'
                                'extern "C" int reads(int M, int K) { return w4a8::reads_in_place(M, K); }\n'
                                'extern "C" int writes(int M, int N, int K) { return w4a8::writes_in_place(M, N, K); }\n')
    subprocess.run(["g++", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "shim.so"), str(d / "shim.cpp")], check=True)
    return ctypes.CDLL(str(d / "shim.so"))


@pytest.fixture(scope="module")
def in_place(shim):
    f = shim.in_place
    f.restype, f.argtypes = ctypes.c_uint64, [ctypes.c_int] + [ctypes.c_uint64] * 5
    return f


def test_whole_buffer_in_one_pinned_range(in_place):
    start, size = 0x7F0000000000, 8192
    for p, n in ((start, 8192), (start + 16, 8176), (start + 4096, 1), (start, 0)):
        assert in_place(1, p, start, size, p, n) == p
    # past the end of the registered part, by a byte and by more than all of it; behind a gap the driver reports another range
    for p, n in ((start, 8193), (start + 16, 8192), (start + 8176, 32), (start + 16, 1 << 63), (start, 2 ** 64 - 1)):
        assert in_place(1, p, start, size, p, n) == 0
    assert in_place(1, start - 16, start, size, start - 16, 16) == 0


def test_what_a_kernel_cannot_address(in_place):
    p = 0x7F0000000000
    assert in_place(0, p, p, 4096, p, 64) == 0               # pageable
    assert in_place(1, 0, p, 4096, p, 64) == 0               # pinned, not mapped
    assert in_place(1, p + 8, p, 4096, p + 8, 64) == 0       # 16-byte accesses would be misaligned
    assert in_place(1, p + 32, p, 0, p, 64) == 0             # no range known
    assert in_place(1, 0x200000, p, 4096, p + 64, 64) == 0x200000      # another address on the device


def test_sizes(shim):
    """Long rows are copied: a CTA that reads one over the bus, twice, is slower than the copy engine."""
    assert shim.reads(64, 4096) and not shim.reads(65, 4096)
    assert shim.reads(1, 32768) and shim.reads(8, 32768) and not shim.reads(1, 32896) and not shim.reads(1, 262144)
    assert shim.writes(8, 32768, 4096) and not shim.writes(9, 32768, 4096) and not shim.writes(1, 128, 65536)
