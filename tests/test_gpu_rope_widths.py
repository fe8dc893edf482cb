"""w4a8_rope_shifted_keys in both forms of its kernel: 16-byte pieces (D a multiple of 16, up to 256, 16-byte-aligned keys)
with heads that do and do not fill a warp's pieces, from 4 Mi elements on, and the 4-byte form otherwise; each the bf16 of the fp64 definition or
its neighbour, out of place and in place."""
import numpy as np
import pytest
import torch

from oracle import streaming as so
from oracle import w4a8_oracle as onp
from paper_2608_12932_b200 import binding as B
from paper_2608_12932_b200 import workload as wl
from tests.gpu_util import bits, t_u16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,H,D,offset", [(262144, 1, 16, 0), (29200, 3, 48, 0), (13109, 5, 64, 0), (1931, 17, 128, 0), (8193, 2, 256, 0),
                                          (5141, 3, 272, 0), (8192, 4, 128, 2), (8191, 4, 128, 0)])
def test_widths_and_alignments(T, H, D, offset):
    rng = np.random.default_rng(T * 100 + D)
    kb = wl.f32_to_bf16_bits((3.0 * rng.standard_normal((T, H, D))).astype(np.float32))
    pos = rng.integers(0, 100000, T).astype(np.int32)
    flat = torch.zeros(T * H * D + 8, dtype=torch.bfloat16, device="cuda")
    k = flat[offset:offset + T * H * D].view(T, H, D)
    k.copy_(t_u16(kb, torch.bfloat16))
    posd = torch.from_numpy(pos).cuda()
    out = bits(B.w4a8_rope_shifted_keys(k, posd, 37, 1e6))
    B.w4a8_rope_shifted_keys(k, posd, 37, 1e6, out=k)
    assert np.array_equal(out, bits(k))
    ref, _ = so.rope_shifted_keys(kb, pos, 37, 1e6)
    kf = np.abs(onp.bf16_bits_to_f64(kb))
    terms = kf[:, :, :D // 2] + kf[:, :, D // 2:]
    # half a bf16 step of the exact result (2^-9) widened to the neighbour (2^-8), plus fp32 errors of the two terms
    bound = 2.0 ** -8 * np.abs(ref) + 1e-6 * np.concatenate([terms, terms], axis=2)
    assert np.all(np.abs(onp.bf16_bits_to_f64(out) - ref) <= bound)


@pytest.mark.parametrize("T,H,D", [(4096, 8, 128), (5461, 3, 256), (16384, 16, 16), (8193, 8, 128), (12000, 11, 64), (5462, 3, 256)])
def test_a_key_does_not_depend_on_the_window_around_it(T, H, D):
    """A window of 4 Mi elements takes the 16-byte form, its parts the 4-byte one: the same bits for the same key."""
    rng = np.random.default_rng(D)
    k = t_u16(wl.f32_to_bf16_bits((3.0 * rng.standard_normal((T, H, D))).astype(np.float32)), torch.bfloat16)
    pos = torch.from_numpy(rng.integers(0, 100000, T).astype(np.int32)).cuda()
    whole = bits(B.w4a8_rope_shifted_keys(k, pos, 37, 1e6))
    for lo, hi in ((0, T // 2), (T // 2, T), (17, 18)):
        part = bits(B.w4a8_rope_shifted_keys(k[lo:hi].contiguous(), pos[lo:hi].contiguous(), 37, 1e6))
        assert np.array_equal(part, whole[lo:hi])
