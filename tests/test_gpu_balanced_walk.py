"""GPU parity of the tensor-core kernels' balanced walk, where tiles are shared by neighbouring CTAs and their sums are
handed over through the workspace: odd group counts, so that ranges begin and end anywhere in a tile, and a ragged last
token tile.  Partials D bit-exact, output within the band of the linear layer on sampled rows of every token tile, residual
form within its own band and in place; each twice, since the hand-over flags have to be back at zero for the next call."""
import numpy as np
import pytest
import torch

from oracle import cfast
from oracle import w4a8_oracle as onp
from paper_2608_12932_b200 import binding as B
from paper_2608_12932_b200 import workload as wl
from tests.gpu_util import DeviceLayer, bits, t_u16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N,tile", [(849, 3200, 4096, 128), (849, 2944, 4096, 208), (20, 2688, 19200, 64), (32, 3200, 19200, 64),
                                        (40, 3200, 19200, 64), (64, 3456, 19200, 64), (588, 3200, 2048, 64)])
def test_tiles_shared_by_neighbours(M, K, N, tile):
    plan = B.w4a8_plan(M, N, K)
    assert plan["family"] == B.PATH_TCGEN05 and plan["tile_m"] == tile and plan["balanced"] == 1
    case = wl.make_layer(K, N, 75 + tile, M)
    layer = DeviceLayer(case, M)
    rng = np.random.default_rng(tile)
    edges = np.arange(0, M, tile)
    rows = np.unique(np.concatenate([edges, edges[1:] - 1, edges + tile // 2, [M - 1], rng.integers(0, M, 8)]))
    rows = rows[rows < M]
    r = cfast.w4a8_linear(case["x"][rows], case["qw"], case["sw"], case["z"], 128, want_partials=True)
    qa, sa, asum = layer.quantize(case["x"])
    y, D = layer.gemm(qa, sa, asum, debug=True)
    assert np.array_equal(D[rows], r["D"])
    ok, ratio = onp.within_tolerance(y[rows], r["ref"])
    assert ok, f"worst |err|/bound = {ratio:.3f}"
    assert np.array_equal(layer.gemm(qa, sa, asum)[0], y)
    r_bits = wl.f32_to_bf16_bits((rng.standard_normal((M, N)) * 4).astype(np.float32))
    res = t_u16(r_bits, torch.bfloat16)
    out = B.w4a8_gemm_residual(qa, sa, asum, layer.packed, res, N, layer.ws)
    B.w4a8_gemm_residual(qa, sa, asum, layer.packed, res, N, layer.ws, out=res)
    B.w4a8_check_status(layer.ws)
    assert np.array_equal(bits(out), bits(res))
    ref = r["ref"] + onp.bf16_bits_to_f64(r_bits[rows])
    assert np.all(np.abs(onp.bf16_bits_to_f64(bits(out)[rows]) - ref) <= onp.residual_tolerance(r["ref"], ref))
