"""The dispatch rules that depend on sizes alone, compiled for the CPU: each at sizes where an earlier rule was measured to pick
a slower kernel or form."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_12932_b200", "csrc")
SMS = 148


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("dispatch_rules")
    (d / "shim.cpp").write_text('#include "dispatch_rules.h"\n'
                                'extern "C" int per_channel_tile_height(int M, int n_tiles, int groups, int sms) {\n'
                                '    return w4a8::per_channel_tile_height(M, n_tiles, groups, sms);\n}\n')
    subprocess.run(["g++", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "shim.so"), str(d / "shim.cpp")], check=True)
    return ctypes.CDLL(str(d / "shim.so"))


@pytest.mark.parametrize("K,N,M,height", [(5120, 7168, 300, 208), (5120, 7168, 416, 208), (5120, 7168, 448, 128), (4096, 4096, 520, 208),
                                          (12288, 4096, 576, 208), (4096, 24576, 100, 128), (4096, 24576, 160, 208),
                                          (13824, 5120, 400, 208), (2048, 12288, 256, 128), (4096, 6144, 1024, 208),
                                          (4096, 6144, 64, 64), (4096, 6144, 128, 64), (256, 256, 1, 64)])
def test_per_channel_tile_height(rules, K, N, M, height):
    assert rules.per_channel_tile_height(M, N // 128, K // 128, SMS) == height
