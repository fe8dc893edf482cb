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
                                '    return w4a8::per_channel_tile_height(M, n_tiles, groups, sms);\n}\n'
                                'extern "C" int silu_cluster_ctas(int M, int K) { return w4a8::silu_cluster_ctas(M, K); }\n')
    subprocess.run(["g++", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "shim.so"), str(d / "shim.cpp")], check=True)
    return ctypes.CDLL(str(d / "shim.so"))


@pytest.mark.parametrize("K,N,M,height", [(5120, 7168, 300, 208), (5120, 7168, 416, 208), (5120, 7168, 448, 128), (4096, 4096, 520, 208),
                                          (12288, 4096, 576, 208), (4096, 24576, 100, 128), (4096, 24576, 160, 208),
                                          (13824, 5120, 400, 208), (2048, 12288, 256, 128), (4096, 6144, 1024, 208),
                                          (4096, 6144, 64, 64), (4096, 6144, 128, 64), (256, 256, 1, 64)])
def test_per_channel_tile_height(rules, K, N, M, height):
    assert rules.per_channel_tile_height(M, N // 128, K // 128, SMS) == height


@pytest.mark.parametrize("M,K,ctas", [(1, 128, 1), (32, 512, 1), (256, 512, 1), (700, 2048, 1), (16, 4096, 1), (16, 5120, 8), (24, 6144, 1),
                                      (24, 8192, 8), (40, 12288, 8), (100, 6144, 1), (100, 12288, 8), (160, 8192, 8), (200, 6144, 1),
                                      (200, 12288, 4), (300, 6144, 1), (512, 12288, 2), (700, 12288, 1), (4096, 12288, 1)])
def test_silu_rows_shared_by_a_cluster(rules, M, K, ctas):
    assert rules.silu_cluster_ctas(M, K) == ctas
