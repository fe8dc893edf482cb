"""GPU parity of the tensor-core kernel's K split at 128- and 208-row tiles where its exchange can go wrong: two to four
slices of equal and unequal length, shares of 13 to 26 runs of four tokens, token counts that end inside a run, inside a
share and before the second half of the drain warps.  Partials D bit-exact, output within the band of the linear layer,
residual form within its own band and equal to the plain one for a zero residual."""
import numpy as np
import pytest
import torch

from oracle import cfast
from oracle import w4a8_oracle as onp
from paper_2608_12932_b200 import binding as B
from paper_2608_12932_b200 import workload as wl
from tests.gpu_util import DeviceLayer, bits, t_u16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,N,tile,slices,Ms", [(13056, 8192, 128, 2, (66, 128)), (5248, 5120, 128, 3, (66, 101, 127)),
                                                (17408, 4096, 128, 4, (65, 98, 128)), (4224, 6144, 208, 2, (193, 207)),
                                                (3200, 5120, 208, 3, (193, 206)), (8448, 4096, 208, 4, (131, 193, 208))])
def test_exchange(K, N, tile, slices, Ms):
    M_max = max(Ms)
    case = wl.make_layer(K, N, 90 + slices, M_max)
    layer = DeviceLayer(case, M_max)
    r = cfast.w4a8_linear(case["x"], case["qw"], case["sw"], case["z"], 128, want_partials=True)
    rng = np.random.default_rng(K)
    r_bits = wl.f32_to_bf16_bits((rng.standard_normal((M_max, N)) * 4).astype(np.float32))
    packed = B.w4a8_pack_weights(torch.from_numpy(case["qw"]).cuda(), t_u16(case["sw"], torch.float16), torch.from_numpy(case["z"]).cuda())
    ws = B.new_workspace(M_max, N, K)
    for M in Ms:
        plan = B.w4a8_plan(M, N, K)
        assert (plan["tile_m"], plan["k_slices"]) == (tile, slices)
        qa, sa, asum = layer.quantize(case["x"][:M])
        y, D = layer.gemm(qa, sa, asum, path=B.PATH_TCGEN05, debug=True)
        assert np.array_equal(D, r["D"][:M])
        ok, ratio = onp.within_tolerance(y, r["ref"][:M])
        assert ok, f"worst |err|/bound = {ratio:.3f}"
        q = B.w4a8_quantize_act(t_u16(case["x"][:M], torch.bfloat16))
        plain = B.w4a8_gemm(*q, packed, N, ws)
        assert np.array_equal(bits(plain), y)
        res = t_u16(r_bits[:M], torch.bfloat16)
        guard = torch.full((M + 4, N), 7.0, dtype=torch.bfloat16, device="cuda")      # rows past M stay as they are
        B.w4a8_gemm_residual(*q, packed, res, N, ws, out=guard[:M])
        B.w4a8_check_status(ws)
        assert bool((guard[M:] == 7.0).all())
        ref = r["ref"][:M] + onp.bf16_bits_to_f64(r_bits[:M])
        err = np.abs(onp.bf16_bits_to_f64(bits(guard[:M])) - ref)
        assert np.all(err <= onp.residual_tolerance(r["ref"][:M], ref))
        zero = B.w4a8_gemm_residual(*q, packed, torch.zeros_like(res), N, ws)
        assert bool((zero == plain).all())
