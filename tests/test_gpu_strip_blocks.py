"""GPU parity of the strip kernel with two token blocks (9 to 16 tokens, one CTA per SM or one per strip) where it can go wrong: fewer strips
than SMs, strips shared by neighbouring CTAs, a ragged last stage, one group, and both sides of the rules that leave a long K
over few channels and a short one over many to the cluster kernel.  Partials D bit-exact, output within the band of the linear layer, residual form
within its own."""
import numpy as np
import pytest
import torch

from oracle import cfast
from oracle import w4a8_oracle as onp
from paper_2608_12932_b200 import binding as B
from paper_2608_12932_b200 import workload as wl
from tests.gpu_util import DeviceLayer, bits, t_u16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,N,family", [(128, 128, B.PATH_STRIP), (2048, 1920, B.PATH_STRIP), (2176, 1920, B.PATH_SPLITK), (512, 5120, B.PATH_SPLITK), (640, 6144, B.PATH_STRIP), (1152, 8192, B.PATH_STRIP),
                                        (2176, 2048, B.PATH_STRIP), (4096, 4096, B.PATH_STRIP), (1152, 5120, B.PATH_STRIP),
                                        (6144, 4864, B.PATH_STRIP)])
def test_two_token_blocks(K, N, family):
    case = wl.make_layer(K, N, 40 + N // 128, 16)
    layer = DeviceLayer(case, 16)
    r = cfast.w4a8_linear(case["x"], case["qw"], case["sw"], case["z"], 128, want_partials=True)
    r_bits = wl.f32_to_bf16_bits((np.random.default_rng(K).standard_normal((16, N)) * 4).astype(np.float32))
    for M in (9, 13, 16):
        assert B.w4a8_plan(M, N, K)["family"] == family
        qa, sa, asum = layer.quantize(case["x"][:M])
        y, D = layer.gemm(qa, sa, asum, debug=True)
        assert np.array_equal(D, r["D"][:M])
        ok, ratio = onp.within_tolerance(y, r["ref"][:M])
        assert ok, f"worst |err|/bound = {ratio:.3f}"
        for _ in range(2):                                      # the hand-over words are back at zero for the second call
            assert np.array_equal(layer.gemm(qa, sa, asum)[0], y)
        res = t_u16(r_bits[:M], torch.bfloat16)
        out = B.w4a8_gemm_residual(qa, sa, asum, layer.packed, res, N, layer.ws)
        B.w4a8_check_status(layer.ws)
        ref = r["ref"][:M] + onp.bf16_bits_to_f64(r_bits[:M])
        assert np.all(np.abs(onp.bf16_bits_to_f64(bits(out)) - ref) <= onp.residual_tolerance(r["ref"][:M], ref))
