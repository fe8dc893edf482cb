"""GPU parity of the short-tile tensor-core kernel (64-row token tiles, cut to 32 columns up to 32 tokens) where it can go
wrong: odd group counts against its two-group steps, one group, both tile widths and their edges, K splits with uneven
shares, more tiles than SMs, and the extreme partials that its accumulator bias has to cover.  Partials D
bit-exact, output within the band of the linear layer, against the CPU oracle."""
import numpy as np
import pytest

from oracle import cfast
from oracle import w4a8_oracle as onp
from paper_2608_12932_b200 import binding as B
from paper_2608_12932_b200 import workload as wl
from tests.gpu_util import DeviceLayer

pytestmark = pytest.mark.gpu


def check(case, layer, M, debug=True):
    qa, sa, asum = layer.quantize(case["x"][:M])
    y, D = layer.gemm(qa, sa, asum, path=B.PATH_TCGEN05, debug=debug)
    r = cfast.w4a8_linear(case["x"][:M], case["qw"], case["sw"], case["z"], 128, want_partials=debug)
    if debug:
        assert np.array_equal(D, r["D"])
    ok, ratio = onp.within_tolerance(y, r["ref"])
    assert ok, f"worst |err|/bound = {ratio:.3f}"
    return y


@pytest.mark.parametrize("K,N", [(128, 128), (256, 256), (384, 128), (512, 256), (640, 384), (1664, 256), (2304, 384)])
def test_group_counts_and_tile_edges(K, N):
    """1, 2, 3, 4, 5, 13 and 18 groups; token counts at the edges of the 16-column MMA steps, of both tiles and of several tiles.  (Up
    to four groups, more than 32 tokens take the 64-row tiles of gemm_tcgen05.cu: their first and last sizes are here too.)"""
    case = wl.make_layer(K, N, 60 + K // 128, 130)
    layer = DeviceLayer(case, 130)
    for M in (1, 15, 16, 17, 31, 32, 33, 47, 48, 49, 63, 64, 65, 127, 128, 129):
        if M > 64:                                          # (up to 64 tokens no taller tile is considered)
            plan = B.w4a8_plan(M, N, K)
            assert plan["family"] == B.PATH_TCGEN05 and plan["tile_m"] == 64
        check(case, layer, M)


@pytest.mark.parametrize("M,K,N", [(20, 3200, 512), (40, 3200, 512), (64, 3456, 512), (100, 3456, 256)])
def test_uneven_k_split(M, K, N):
    """25 or 27 groups over two to four slices: uneven shares, odd and even, and tokens that do not fill the dealt-out runs."""
    case = wl.make_layer(K, N, 71, M)
    layer = DeviceLayer(case, M)
    if M > 32:                                              # (at 20 tokens the dispatch takes the cluster kernel: forced here)
        plan = B.w4a8_plan(M, N, K)
        assert plan["family"] == B.PATH_TCGEN05 and plan["tile_m"] == 64 and plan["k_slices"] > 1
    y = check(case, layer, M)
    assert np.array_equal(y, check(case, layer, M, debug=False))


@pytest.mark.parametrize("M,K,N", [(20, 1152, 24576), (40, 1152, 24576), (130, 1152, 24576)])
def test_more_tiles_than_sms(M, K, N):
    """More tiles than SMs, nine groups each, as whole tiles: rings and accumulator buffers run on from one tile to the next
    behind a lone last group.  (Tiles shared by neighbouring CTAs: test_gpu_balanced_walk.py.)"""
    case = wl.make_layer(K, N, 72, M)
    layer = DeviceLayer(case, M)
    plan = B.w4a8_plan(M, N, K)
    assert plan["tile_m"] == 64 and plan["k_slices"] == 1 and plan["balanced"] == 0
    y1 = check(case, layer, M, debug=False)
    assert np.array_equal(y1, check(case, layer, M, debug=False))


@pytest.mark.parametrize("M,K", [(17, 384), (64, 384), (33, 640), (64, 640)])
def test_extreme_partials(M, K):
    """Codes and zero points at the ends of their ranges against activation codes at +-127: |D| = 243840, the bias is 245760."""
    rng = np.random.default_rng(5)
    N = 256
    case = wl.random_codes(rng, M, N, K)
    case["qw"][:] = np.where(rng.integers(0, 2, (N, 1)) == 1, 15, 0)
    case["z"][:] = np.where(case["qw"][:, 0] == 15, 0, 15)[None, :]
    sign = np.where(rng.integers(0, 2, (M, 1)) == 1, 1.0, -1.0)
    case["x"] = wl.f32_to_bf16_bits((sign * np.ones((M, K))).astype(np.float32))
    layer = DeviceLayer(case, M)
    check(case, layer, M)
    qa, sa, asum = layer.quantize(case["x"])
    _, D = layer.gemm(qa, sa, asum, path=B.PATH_TCGEN05, debug=True)
    assert np.abs(D).max() == 15 * 127 * 128
