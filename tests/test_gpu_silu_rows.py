"""GPU parity of w4a8_silu_mul_quantize where its form changes: a row shared by a cluster of eight, four or two CTAs (few
rows), by one (many rows), at channel counts that share out unevenly.  h against the oracle on the same gate and up values
(one bf16 step at most), scales, codes and group sums bit-exact on the kernel's own h."""
import numpy as np
import pytest
import torch

from oracle import w4a8_oracle as onp
from paper_2608_12932_b200 import binding as B
from paper_2608_12932_b200 import workload as wl
from tests.gpu_util import bits, t_u16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,I", [(1, 128), (17, 384), (32, 13824), (33, 1152), (160, 6144), (161, 6144), (256, 2176), (257, 12288),
                                 (700, 1280), (701, 1280), (40, 25600), (1, 5120), (16, 5248), (17, 8192), (32, 28672), (33, 5120),
                                 (48, 13824), (49, 8320), (65, 12288), (128, 12416), (129, 8192), (160, 16384), (160, 16512), (161, 8192),
                                 (256, 10368), (257, 10240), (600, 10240), (601, 10240)])
def test_rows_and_channel_shares(M, I):
    rng = np.random.default_rng(M + I)
    y = wl.f32_to_bf16_bits((rng.standard_normal((M, 2 * I)) * 2).astype(np.float32))
    y[M // 2] = 0                                               # a row of zeros: scale 0, codes 0
    h, qa, sa, asum = B.w4a8_silu_mul_quantize(t_u16(y, torch.bfloat16))
    torch.cuda.synchronize()
    hb = bits(h)
    runs = y.reshape(M, I // 8, 2, 8)
    gate, up = runs[:, :, 0].reshape(M, I), runs[:, :, 1].reshape(M, I)
    ref, _ = onp.silu_mul(gate, up)
    err = np.abs(onp.bf16_bits_to_f64(hb) - ref)
    assert np.all(err <= 2.0 ** -7 * np.abs(ref) + 1e-30)        # half a step of the reference plus one step of the kernel
    qa_o, sa_o, asum_o = onp.quantize_act(hb, 128)
    assert np.array_equal(bits(sa), sa_o) and np.array_equal(qa.cpu().numpy(), qa_o) and np.array_equal(asum.cpu().numpy(), asum_o)
